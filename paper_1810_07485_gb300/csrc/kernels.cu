// Kernels of one continuous-time loop-cluster update (Sec. 2 MC step, Sec. 3.2
// union-find), batched over independent chains.  Work is cut into tiles of 128
// consecutive cells (bond x time window) of one chain; a tile is one block.
//
// Phase order per update (the Sec. 4.3 cost table's rows in brackets):
//   k_start          spin parity of every bond at each time-block start; scratch
//                    reset
//   k_insert         per cell: Poisson candidates, keep the antiparallel ones,
//                    merge with old operators, write vertices; offsets by
//                    decoupled look-back over the tiles          [1, 2]
//   k_cut            last leg per subsite, tau=0 subspin permutation
//   k_link           predecessor of each leg on both subsites; union of the two
//                    fragments below each vertex (lock-free, min root)    [2]
//   k_compress       root of every node, one coin per loop              [3]
//   k_est            new operator flags, loop lengths (tile-local loops in
//                    shared memory, others in global accumulators)      [4]
//   k_scan_ops       operator offsets per tile (chains of many tiles)
//   k_compact        next operator list, squared lengths of open loops  [8]
//   k_sites          spins at tau = 0, vertex-free loops (chains of few
//                    tiles: blocks of k_compact's launch)               [8]
//   k_final          per-chain record, running sums, buffer swap
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <mutex>

#include "dev.cuh"
#include "kernels.h"
#include "uf.cuh"

namespace lcq {

__constant__ uint64_t c_T_full[KMAX];
// exp(i 2 pi k / 2^16) in units of 2^-30, k = 0..2^16 (temporal moment)
__device__ int2 g_phase_tab[(1 << PHASE_BITS) + 1];

// ---- block-wide helpers (blockDim.x is a multiple of 32, <= 1024) ---------
template <typename T>
__device__ T warp_incl_scan(T v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

template <typename T>
__device__ T block_excl_scan(T v, T *sm, T &total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  T inc = warp_incl_scan(v);
  if (lane == 31) sm[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    T x = (lane < nw) ? sm[lane] : T(0);
    T xi = warp_incl_scan(x);
    if (lane < nw) sm[lane] = xi - x;
    if (lane == nw - 1) sm[32] = xi;
  }
  __syncthreads();
  T res = sm[wid] + inc - v;
  total = sm[32];
  __syncthreads();
  return res;
}

template <typename T>
__device__ T block_sum(T v, T *sm) {
  T tot;
  block_excl_scan(v, sm, tot);
  return tot;
}

__device__ __forceinline__ u128 shfl_down_u128(u128 v, int o) {
  const unsigned long long l = __shfl_down_sync(0xffffffffu, (unsigned long long)v, o);
  const unsigned long long h = __shfl_down_sync(0xffffffffu, (unsigned long long)(v >> 64), o);
  return ((u128)h << 64) | (u128)l;
}

// Exact sum of a 128-bit value over the warp, on every lane: eight warp
// reductions of 16-bit pieces (32 of them stay below 2^21) instead of five
// rounds of four shuffles and a 128-bit add.
__device__ __forceinline__ u128 warp_sum_u128(u128 v) {
  u128 t = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint32_t w = (uint32_t)(v >> (32 * k));
    const uint32_t lo = __reduce_add_sync(0xffffffffu, w & 0xffffu), hi = __reduce_add_sync(0xffffffffu, w >> 16);
    t += (u128)(lo + ((unsigned long long)hi << 16)) << (32 * k);
  }
  return t;
}

// Exact block-wide sums of one count (block total below 2^32) and two (Z: three)
// 128-bit values with a single barrier; the totals are valid in thread 0.  Once
// per kernel.
template <bool Z, bool SPARSE = false>
__device__ void block_sums(long long &c, u128 &x, u128 &y, u128 &z) {
  __shared__ uint32_t pc[32];
  __shared__ u128 px[32], py[32], pz[Z ? 32 : 1];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint32_t n = __reduce_add_sync(0xffffffffu, (uint32_t)c);
  if (!SPARSE || __any_sync(0xffffffffu, (x | y | z) != 0)) {
    x = warp_sum_u128(x);
    y = warp_sum_u128(y);
    if (Z) z = warp_sum_u128(z);
  }
  if (lane == 0) {
    pc[wid] = n;
    px[wid] = x;
    py[wid] = y;
    if (Z) pz[wid] = z;
  }
  __syncthreads();
  if (wid == 0) {
    c = __reduce_add_sync(0xffffffffu, lane < nw ? pc[lane] : 0u);
    x = warp_sum_u128(lane < nw ? px[lane] : (u128)0);
    y = warp_sum_u128(lane < nw ? py[lane] : (u128)0);
    if (Z) z = warp_sum_u128(lane < nw ? pz[lane] : (u128)0);
  }
}

// Whether the update has stopped.  The status word may be set while a launch's
// blocks start: by the launch itself (a chain without room, a wait that ran out,
// a failed check) and by the kernels of another spin group, which run beside it.
// Threads that read it one by one may then disagree, and the ones that go on would
// use shared memory that the others never wrote.  So a kernel whose threads work
// together takes one answer for the block (a warp, where a warp works alone), at its
// first barrier where it can: what comes before reads and writes nothing that the
// cells' offsets could lead out of bounds, and the word is on its way meanwhile.  One
// thread reads it for the block (a reduction over the barrier took 1 to 2 % of an
// update of few tiles: L=1024 77.7 against 75.8 us, S = 3/2, 288 tiles, 137 / 133.5).
// The answer of a single thread is enough where nothing that can set the word runs
// beside the launch (k_start, k_compact, k_sites, k_final) or each thread works alone
// (k_check_forest).
__device__ __forceinline__ bool halted(const Scratch &s) { return __ldcg(s.status) != 0; }
__device__ __forceinline__ bool halted_warp(const Scratch &s) { return __any_sync(0xffffffffu, halted(s)); }
__device__ __forceinline__ bool halted_block(const Scratch &s) { return __syncthreads_or(halted(s)) != 0; }

// Tile blocks of the vertex-parallel kernels: TPB threads walk the tile's
// vertices in id order (coalesced).  A launch of few tiles leaves most of the
// SMs' warp slots empty and its time is the longest tile's chain of steps:
// there linking, compression and loop properties take TPB_WIDE threads per tile
// while two such blocks per SM hold every tile.  One update, us, 256 / 1024
// threads: S = 1/2, 2 tiles 94 / 74, 152 tiles 117 / 93, 301 tiles 129 / 110,
// 598 tiles 146 / 149; S = 2, 68 tiles 207 / 166, 294 tiles 254 / 209.
constexpr int TPB = 256, TPB_WIDE = 1024;
constexpr int64_t WIDE_TILES = 152 * 2;

// A value that every lane holds, in a form the compiler knows to be uniform
// (loops bounded by it need no divergence handling).
__device__ __forceinline__ int uniform(int x) { return (int)__reduce_max_sync(0xffffffffu, x); }

__device__ __forceinline__ uint32_t uniform(uint32_t x) { return __reduce_max_sync(0xffffffffu, x); }

// Vertex bitmaps are written a word (32 vertices) at a time by the warp that
// handles them; a tile's first and last words are shared with its neighbours
// and take an atomic (the bitmap starts the update at zero).
__device__ __forceinline__ void store_word(uint32_t *bits, int64_t word, uint32_t x, int v0, int a, int e) {
  if (v0 >= a && v0 + 32 <= e)
    bits[word] = x;
  else if (x)
    atomicOr(bits + word, x);
}

// ---- start of an update: bond parities, scratch reset --------------------------
// bpar[(blk) * nbond + b] = parity of the operators of bond b in time blocks
// before blk; row nblk is the parity over the whole period.
__device__ __forceinline__ void bond_parity(const DevChain &C, int b, const Scratch &s) {
  const int32_t *op = C.op_ptr[C.cur];
  uint8_t *row = s.bpar + C.bpar_off;
  uint8_t p = 0;
  row[b] = 0;
  for (int blk = 0; blk < C.nblk; ++blk) {
    int j0 = blk * TW;
    int tw = min(TW, C.nwin - j0);
    int c0 = blk * C.nbond * TW + b * tw;
    p ^= (uint8_t)((op[c0 + tw] - op[c0]) & 1);
    row[(int64_t)(blk + 1) * C.nbond + b] = p;
  }
}

// The first nbb blocks take a block of bonds each; the others reset the
// insertion's look-back words and tile tickets, the operator scan's part words
// and the five per-vertex bitmaps (open marks, open roots, flips, new
// operators, crossing marks), which start each update at zero.  One launch for
// both: a small chain's update is a chain of short launches.
__global__ void __launch_bounds__(BOND_BLOCK) k_start(const DevChain *__restrict__ ch,
                                                      const int2 *__restrict__ tab, int64_t nbb, Scratch s,
                                                      int64_t ntile, int64_t nw) {
  if (blockIdx.x < nbb) {
    if (halted(s)) return;
    const int2 t = tab[blockIdx.x];
    const int b = t.y * BOND_BLOCK + threadIdx.x;
    if (b < ch[t.x].nbond) bond_parity(ch[t.x], b, s);
    return;
  }
  const int64_t i0 = (blockIdx.x - nbb) * blockDim.x + threadIdx.x;
  const int64_t step = (gridDim.x - nbb) * blockDim.x;
  for (int64_t i = i0; i < nw; i += step) {
    s.openmark[i] = 0u;
    s.openroot[i] = 0u;
    s.flipbits[i] = 0u;
    s.newbits[i] = 0u;
    s.xmark[i] = 0u;
  }
  for (int64_t i = i0; i < ntile; i += step) s.tile_state[i] = 0ull;
  for (int64_t i = i0; i < SCAN_PARTS; i += step) s.part_state[i] = 0ull;
  if (i0 < QMAX) s.tickets[i0] = 0u;
}

// ---- insertion (labeling, rules i-iii) --------------------------------------
// Imaginary times are handled as the int64 bit patterns of non-negative doubles
// (same order as the values); the one fp64 instruction per candidate is the fused
// multiply-add of its time, fma(t_end - t0, u, t0).
// Single pass: every tile counts its cells' vertices, publishes the count, and
// gets the chain-local offset of its first vertex by decoupled look-back over
// the tiles before it (tile order = order in which blocks took their ticket,
// so every tile waited on has started and publishes its count without
// waiting).  Each wait is bounded; it also gives up when the update halts.
constexpr unsigned long long LB_AGG = 1ull, LB_INC = 2ull, LB_MASK = (1ull << 62) - 1;
constexpr int LB_MAX_SPINS = 1 << 24;

__device__ __forceinline__ void lb_publish(unsigned long long *st, int64_t g, unsigned long long flag,
                                           int64_t v) {
  atomicExch(st + g, (flag << 62) | ((unsigned long long)v & LB_MASK));
}

// Warp-cooperative look-back (run by warp 0): lane l inspects tile g-1-l of a
// window of 32 predecessors; the window moves down until it holds a tile with
// an inclusive prefix.  first = the chain's first tile, which publishes its
// inclusive prefix at once, so the walk never leaves the chain.
__device__ int64_t lb_lookback(unsigned long long *st, int64_t g, int64_t first, const Scratch &s) {
  const int lane = threadIdx.x & 31;
  int64_t excl = 0;
  int spins = 0;
  for (int64_t p = g - 1;;) {
    const int64_t idx = p - lane;
    unsigned long long x = (LB_INC << 62);  // below the chain: inclusive 0
    if (idx >= first) x = *((volatile unsigned long long *)(st + idx));
    const unsigned long long f = x >> 62;
    const unsigned inc = __ballot_sync(0xffffffffu, f == LB_INC);
    const unsigned none = __ballot_sync(0xffffffffu, f == 0);
    const int k = inc ? __ffs(inc) - 1 : 31;  // lanes 0..k are summed
    if (none & (k == 31 ? 0xffffffffu : ((2u << k) - 1u))) {  // a tile up to lane k not ready
      if (++spins > LB_MAX_SPINS) {
        if (lane == 0) atomicOr(s.status, ST_TIMEOUT);
        return 0;
      }
      if ((spins & 255) == 0 && halted_warp(s)) return 0;
      __nanosleep(32);
      continue;
    }
    long long v = (lane <= k) ? (long long)(x & LB_MASK) : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    excl += v;
    if (inc) return excl;
    p -= 32;
  }
}

// Candidate-parallel insertion, a warp for every 16 (or 8) cells of the tile.
// Lanes l and l + 16 (l + 8) set up cell l together: each takes the neighbour bonds of one of
// the cell's subsites (operator ranges, spin parity at the window start) and
// one of the cell's first two Philox calls (call 0 gives the number K of
// candidates and candidate 0, call m >= 1 candidates 2m-1 and 2m).  The
// remaining calls are spread over the lanes, then the candidates: each lane
// forms a candidate's time, takes the antiparallel test, and the kept ones
// are packed in place by ballots, so that a cell's kept candidates stay
// contiguous.  A kept candidate's place inside its cell follows from ranks:
// among the kept candidates by (u53, draw index), and against the old operators
// by time (an old operator goes first on a tie).  It marks its position; the
// unmarked positions are the old operators in their order, so the warp writes
// its vertices in id order (time, flag, cell; the parent forest is set by the
// linking kernels).
//
// The kernel is bound by instruction issue (85 % of the issue slots; 26 of 32
// lanes active).  Warps work on their own cells, so that the block meets only
// for the offsets, and packed candidates and marked positions leave no lane
// walking a list alone: 1.04 -> 0.78 ms at L=16384, beta=4096 (4.65e7
// vertices), against one thread per cell for the set-up with block-wide scans
// and lists (eleven barriers, issue 65 %).  Of the 0.78 ms the set-up takes
// 0.16, the draws 0.08, the decisions 0.22, the places 0.20, the look-back 0.02
// and the writes 0.13.  Six blocks per SM at 40 registers (five at 48: 0.82).
// A warp stages InsWarp::CAP candidates (mean 128 for 16 cells, sigma 11): one whose cells have
// more runs them in groups, counting in a first pass and drawing again in the
// writing pass.
//
// NW warps per tile: 8, or 16 with 8 cells each for launches of few tiles, whose
// time is one tile's chain of steps (insertion in us, 8 / 16 warps: L=64 20.6 /
// 18.0, L=1024, 128 tiles, 28.9 / 21.3, S = 2, 65 tiles, 36 / 29).  There lanes
// l + 16 and l + 24 repeat what l and l + 8 do in the set-up.
constexpr int INS_WARPS = 8, INS_WARPS_WIDE = 16;
template <int NW>
struct InsWarp {
  static constexpr int WC = TILE / NW;  // cells of a warp
  // candidates a warp stages, and vertices a group of its cells may have for
  // their positions to be marked in shared memory (mean 177 for 16 cells of a
  // thermalized S = 1/2 chain, sigma 15)
  static constexpr int CAP = NW == 8 ? 168 : 104, MARKS = NW == 8 ? 288 : 160;
  static_assert(WC <= 16, "two lanes per cell, four bits of a key");
  static_assert(CAP >= KMAX - 1, "a cell's candidates fit");
};
// The lanes that move their cell's staged ranges (the neighbours' of their side):
// one per cell and side, since a range is moved in place and a lane that repeats
// another would move it a second time.  With 8 cells lanes 16 to 31 repeat.
template <int NW>
__host__ __device__ constexpr bool ins_moves(int lane) {
  return lane < 2 * InsWarp<NW>::WC;
}
template <int NW>
constexpr bool ins_moves_once() {
  int n[2][InsWarp<NW>::WC] = {};
  for (int l = 0; l < 32; ++l)
    if (ins_moves<NW>(l)) ++n[(l / InsWarp<NW>::WC) & 1][l & (InsWarp<NW>::WC - 1)];
  for (int c = 0; c < InsWarp<NW>::WC; ++c)
    if (n[0][c] != 1 || n[1][c] != 1) return false;
  return true;
}
static_assert(ins_moves_once<INS_WARPS>() && ins_moves_once<INS_WARPS_WIDE>(), "each range is moved once");

constexpr int INS_MIN_SPAN = 256;  // smallest group a chain may ask for (tests), in candidates of a whole tile

// Old operator times a tile stages in shared memory: its own cells' and those
// of the cells up to 8 Q^2 cells away (the neighbour bonds of the same
// windows), when they fit (about 1230 for a thermalized S = 1 tile).
template <int Q>
struct InsStage {
  static constexpr int N = Q == 1 ? 896 : (Q == 2 ? 1536 : 2048);
  static constexpr int PAD = 4;  // entries a search may read past the last one
};

template <int Q, int NW>
struct InsSmem : InsWarp<NW> {
  using W = InsWarp<NW>;
  static constexpr int NB = 4 * Q - 2;  // neighbour bonds of a cell
  long long sop[InsStage<Q>::N + InsStage<Q>::PAD];  // staged old operator times (16-byte aligned: first member)
  // Per warp: the candidates' keys (cell in the warp << 59 | u53 << 6 | draw
  // index), then, for the kept ones, the same and the times' bits.  Two more
  // entries: a sentinel, and the second half of a pair load.
  unsigned long long key[NW][W::CAP + 2];
  long long tau[NW][W::CAP];
  // Per cell: neighbour and own operator ranges (from the first staged operator
  // if all of the warp's ranges are staged), window, kept candidates
  int2 nb[TILE][NB], own[TILE];
  int j[TILE], cex[TILE];
  unsigned short less[TILE], kf[TILE], nk[TILE];  // bit k of less: neighbour bond k < the cell's bond
  // Per warp: a vertex position's kept candidate + 1, 0 for an old operator
  uint8_t mark[NW][W::MARKS];
  uint8_t par0[TILE];
  unsigned long long T[2][KMAX];  // Poisson thresholds: full windows, last window
  int wtot[NW];
  int slo, shi;
  uint64_t bar;
  int64_t excl;
  int64_t gt;
};

static_assert(sizeof(InsSmem<1, INS_WARPS>) <= 228 * 1024 / 6 - 1024, "six blocks per SM");

// Number of times below thr in t[lo, hi) (ascending).  ST (staged operators):
// the ranges hold 4.7 operators on average; more than 7 are halved first, then
// three steps follow without branches, each reading up to PAD - 1 entries past
// hi (a halving loop took twice the instructions).
template <bool ST>
__device__ __forceinline__ int times_below(const long long *t, int lo, int hi, long long thr) {
  const int base = lo;
  while (hi - lo > (ST ? 7 : 0)) {
    const int mid = lo + ((hi - lo) >> 1);  // no overflow near 2^31
    if (t[mid] < thr)
      lo = mid + 1;
    else
      hi = mid;
  }
  if (ST) {
#pragma unroll
    for (int d = 4; d > 0; d >>= 1) {
      const bool in = lo + d <= hi, below = t[lo + d - 1] < thr;
      lo += (in & below) ? d : 0;
    }
  }
  return lo - base;
}

// The double u53 2^-53 of a candidate's key (its bits; unit_bits without the
// case of fewer than 33 significant bits, which is left to it).
__device__ __forceinline__ double key_unit(unsigned long long key) {
  const uint32_t hi = (uint32_t)(key >> 38) & 0x1fffffu, lo = (uint32_t)(key >> 6);
  uint64_t bits;
  if (hi) {  // u53 in [2^(52-s), 2^(53-s)), s < 21
    const int sh = __clz((int)hi) - 11;
    const uint32_t h = __funnelshift_l(lo, hi, sh) + ((uint32_t)(1021 - sh) << 20);
    bits = ((uint64_t)h << 32) | (lo << sh);
  } else {
    bits = unit_bits(lo);
  }
  return __longlong_as_double((long long)bits);
}

// A warp's cells: lanes l and l + WC hold cell l.
struct InsCell {
  int b, j, K, kpre;  // bond, window, candidates, candidates of the cells before it
};

// Times, antiparallel tests and packing of the warp's ns staged candidates;
// returns how many are kept.  ST: every operator range is staged (shared
// memory loads), else ot is the chain's operator list.  A candidate's time is
// tau = fma(d, u53 2^-53, t0) (one IEEE fused multiply-add); it is kept if its
// bond's spins are antiparallel there (parity at the window start flipped by
// the neighbour operators before it; order (time, bond)).
template <int Q, int NW, bool ST>
__device__ __forceinline__ int ins_decide(const DevChain &C, InsSmem<Q, NW> &S, const long long *otau, int wid,
                                          int ns) {
  constexpr int WC = InsWarp<NW>::WC;
  const int lane = threadIdx.x & 31;
  const long long *ot = ST ? S.sop : otau;
  int nkept = 0;
  for (int i0 = 0; i0 < ns; i0 += 32) {
    const int slot = i0 + lane;
    bool keep = false;
    unsigned long long key = 1;
    long long tau = 0;
    int c = 0;
    if (slot < ns) {
      key = S.key[wid][slot];
      c = (int)(key >> 59);
      const int cw = wid * WC + c;
      const uint64_t *win = C.win + 3 * S.j[cw];
      const double t0 = __longlong_as_double((long long)win[0]);
      const long long teb = (long long)win[1];
      const double d = __longlong_as_double((long long)win[2]);
      tau = __double_as_longlong(__fma_rn(d, key_unit(key), t0));
      if (tau < teb) {
        int p = S.par0[cw];
        const int less = S.less[cw];
#pragma unroll
        for (int k = 0; k < InsSmem<Q, NW>::NB; ++k) {
          const int2 r = S.nb[cw][k];
          p ^= times_below<ST>(ot, r.x, r.y, tau + ((less >> k) & 1));
        }
        keep = p & 1;
      }
    }
    const unsigned km = __ballot_sync(0xffffffffu, keep);
    const int at = nkept + __popc(km & ((1u << lane) - 1u));
    __syncwarp();  // every lane has read its candidate: pack over the ones read
    if (slot < ns && (key & 63) == 0) S.kf[wid * WC + c] = (unsigned short)at;
    if (keep) {
      S.key[wid][at] = key;
      S.tau[wid][at] = tau;
    }
    nkept += __popc(km);
  }
  __syncwarp();
  if (lane == 0) S.key[wid][nkept] = ~0ull;
  return nkept;
}

// Draw and decide the candidates of the warp's cells [c0, c1); o: the lane's
// output of Philox call (lane >= 16) of its cell.  Sets kf and nk of the cells;
// returns the number kept.
template <int Q, int NW>
__device__ __forceinline__ int ins_group(const DevChain &C, InsSmem<Q, NW> &S, const long long *otau, int wid,
                                         const InsCell &X, const U4 &o, int c0, int c1, bool staged, uint32_t sweep,
                                         uint32_t k0, uint32_t k1) {
  constexpr int WC = InsWarp<NW>::WC;
  const int lane = threadIdx.x & 31, cl = lane & (WC - 1), side = (lane / WC) & 1;
  const bool in = cl >= c0 && cl < c1;
  const int kb = __shfl_sync(0xffffffffu, X.kpre, c0);
  const int ns = uniform(__shfl_sync(0xffffffffu, X.kpre + X.K, c1 - 1) - kb);
  auto put = [&](int c, int slot, int k, uint32_t lo, uint32_t hi) {
    const uint64_t u53 = ((uint64_t)lo | ((uint64_t)hi << 32)) >> 11;
    S.key[wid][slot] = ((uint64_t)c << 59) | (u53 << 6) | (uint64_t)k;
  };
  // calls 0 (lower lanes: candidate 0) and 1 (upper lanes: candidates 1, 2)
  if (in) {
    const int ks = X.kpre - kb;
    if (side && X.K > 1) put(cl, ks + 1, 1, o.x, o.y);
    if (X.K > 2 * side) put(cl, ks + 2 * side, 2 * side, o.z, o.w);
  }
  // calls 2 .. K/2
  const int P = (in && X.K > 3) ? X.K / 2 - 1 : 0;
  int pin = P;  // inclusive scan over the cells (both halves alike)
#pragma unroll
  for (int d = 1; d < WC; d <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, pin, d, WC);
    if (cl >= d) pin += y;
  }
  const int nu = uniform(__shfl_sync(0xffffffffu, pin, WC - 1));
  for (int u0 = 0; u0 < nu; u0 += 32) {
    const int u = u0 + lane;
    int c = 0;  // cells whose calls all come before call u
#pragma unroll
    for (int d = WC / 2; d > 0; d >>= 1) {
      const int y = __shfl_sync(0xffffffffu, pin, c + d - 1);
      if (y <= u) c += d;
    }
    // (for u >= nu the search ends at cell 15; those lanes draw nothing)
    const int first = __shfl_sync(0xffffffffu, pin - P, c), b = __shfl_sync(0xffffffffu, X.b, c);
    const int j = __shfl_sync(0xffffffffu, X.j, c), K = __shfl_sync(0xffffffffu, X.K, c);
    const int ks = __shfl_sync(0xffffffffu, X.kpre, c) - kb;
    if (u < nu) {
      const int m = 2 + u - first, k = 2 * m - 1;
      const U4 p = philox((TAG_INSERT << 24) | (uint32_t)m, (uint32_t)b, (uint32_t)j, sweep, k0, k1);
      if (k < K) put(c, ks + k, k, p.x, p.y);
      if (k + 1 < K) put(c, ks + k + 1, k + 1, p.z, p.w);
    }
  }
  __syncwarp();
  const int nkept = staged ? ins_decide<Q, NW, true>(C, S, otau, wid, ns) : ins_decide<Q, NW, false>(C, S, otau, wid, ns);
  // first kept candidate and number kept per cell; a cell without candidates
  // starts where the next one with candidates does
  const unsigned has = __ballot_sync(0xffffffffu, in && lane < WC && X.K > 0);
  const unsigned from = has >> cl;
  const int nx = from ? cl + __ffs(from) - 1 : cl;
  int kf = (in && X.K > 0) ? S.kf[wid * WC + cl] : nkept;
  kf = __shfl_sync(0xffffffffu, kf, nx);
  const int kn = __shfl_down_sync(0xffffffffu, kf, 1, WC);
  __syncwarp();
  if (in && lane < WC) {
    S.kf[wid * WC + cl] = (unsigned short)kf;
    S.nk[wid * WC + cl] = (unsigned short)((cl == c1 - 1 ? nkept : kn) - kf);
  }
  __syncwarp();
  return nkept;
}

// Positions of the warp's nkept kept candidates among the vertices of its cells
// (cell order, then time): marked in shared memory from position `from` on, or,
// for DIRECT, written to the vertex arrays at once.
template <int Q, int NW, bool ST, bool DIRECT>
__device__ __forceinline__ void ins_place(const DevChain &C, InsSmem<Q, NW> &S, const long long *otau, int wid,
                                          int nkept, int from, int64_t base, const Scratch &s) {
  constexpr int WC = InsWarp<NW>::WC;
  const int lane = threadIdx.x & 31;
  const long long *ot = ST ? S.sop : otau;
  for (int i0 = 0; i0 < nkept; i0 += 32) {
    const int i = i0 + lane;
    if (i < nkept) {
      const unsigned long long key = S.key[wid][i];
      const long long tau = S.tau[wid][i];
      const int cw = wid * WC + (int)(key >> 59);
      // kept candidates ahead, two keys a step from an even place on (one of
      // the cell before is below the cell's keys, what follows is above them)
      const int kf = S.kf[cw], k0 = kf & ~1, k1 = kf + S.nk[cw];
      int r = k0 - kf;
      for (int x = k0; x < k1; x += 2) {
        const ulonglong2 kk = *(const ulonglong2 *)&S.key[wid][x];
        r += (int)(kk.x < key) + (int)(kk.y < key);
      }
      const int2 own = S.own[cw];
      r += times_below<ST>(ot, own.x, own.y, tau + 1);  // old operators at or before tau
      const int pos = S.cex[cw] + r;
      if (DIRECT) {
        const int64_t v = C.vtx_base + base + pos;
        ((long long *)s.vtau)[v] = tau;
        s.vflag[v] = 0;
        s.vcell[v] = (uint8_t)cw;
      } else {
        S.mark[wid][pos - from] = (uint8_t)(i + 1);
      }
    }
    __syncwarp();
  }
}

// Write the marked vertices [0, n) from tile position `from` on, in id order:
// the positions without a mark are the old operators from qa on, in their
// order.  ce: first position of the lane's cell.
template <int Q, int NW, bool ST>
__device__ __forceinline__ void ins_write(const DevChain &C, InsSmem<Q, NW> &S, const long long *otau, int wid, int n,
                                          int from, int ce, int qa, int64_t base, const Scratch &s) {
  constexpr int WC = InsWarp<NW>::WC;
  const int lane = threadIdx.x & 31;
  const int64_t vb = C.vtx_base + base + from;
  long long *vt = (long long *)s.vtau + vb;
  uint8_t *vf = s.vflag + vb, *vc = s.vcell + vb;
  const long long *ot = ST ? S.sop - S.slo : otau;
  for (int i0 = 0; i0 < n; i0 += 32) {
    const int i = i0 + lane, m = i < n ? S.mark[wid][i] : 0;
    const unsigned old = __ballot_sync(0xffffffffu, i < n && m == 0);
    int c = 0;  // largest cell with first position <= i
#pragma unroll
    for (int d = WC / 2; d > 0; d >>= 1) {
      const int y = __shfl_sync(0xffffffffu, ce, c + d);
      if (y <= from + i) c += d;
    }
    if (i < n) {
      vt[i] = m ? S.tau[wid][m - 1] : ot[qa + __popc(old & ((1u << lane) - 1u))];
      vf[i] = m ? 0 : VF_OLD;
      vc[i] = (uint8_t)(wid * WC + c);
    }
    qa += __popc(old);
  }
  __syncwarp();
}

// The old operators [qa, qb) of a group of cells with too many vertices for the
// marks: each finds its place by the kept candidates before it.  q0, ce: first
// operator and first position of the lane's cell.
template <int Q, int NW>
__device__ __noinline__ void ins_write_old(InsSmem<Q, NW> &S, const long long *otau, int wid, int q0, int ce, int qa,
                                           int qb, long long *vt, uint8_t *vf, uint8_t *vc) {
  constexpr int WC = InsWarp<NW>::WC;
  const int lane = threadIdx.x & 31;
  for (int qq = qa; qq < qb; qq += 32) {
    const int q = qq + lane;
    int c = 0;  // largest cell with first operator <= q
#pragma unroll
    for (int d = WC / 2; d > 0; d >>= 1) {
      const int y = __shfl_sync(0xffffffffu, q0, c + d);
      if (y <= q) c += d;
    }
    const int qc = __shfl_sync(0xffffffffu, q0, c), pc = __shfl_sync(0xffffffffu, ce, c);
    if (q < qb) {
      const int cw = wid * WC + c;
      const long long t = otau[q];
      const long long *tt = &S.tau[wid][S.kf[cw]];
      const int n = S.nk[cw];
      int r = q - qc;
      for (int x = 0; x < n; ++x) r += tt[x] < t;
      vt[pc + r] = t;
      vf[pc + r] = VF_OLD;
      vc[pc + r] = (uint8_t)cw;
    }
    __syncwarp();
  }
}

template <int Q, int NW>
__device__ __forceinline__ void insert_tile(InsSmem<Q, NW> &S, DevChain *__restrict__ ch,
                                            const int2 *__restrict__ tab, int64_t blk0, int group,
                                            Scratch s);

// Dynamic shared memory: 36 KB for Q = 1 (six blocks per SM), above the 48 KB
// static limit for the larger neighbour tables and operator stages of Q >= 3.
template <int Q, int NW>
__global__ void __launch_bounds__(32 * NW, NW > 8 ? 2 : (Q == 1 ? 6 : 4)) k_insert(DevChain *__restrict__ ch,
                                                 const int2 *__restrict__ tab, int64_t blk0,
                                                 int group, Scratch s) {
  extern __shared__ __align__(16) unsigned char ins_dyn[];
  insert_tile<Q, NW>(*reinterpret_cast<InsSmem<Q, NW> *>(ins_dyn), ch, tab, blk0, group, s);
}

template <int Q, int NW>
__device__ __forceinline__ void insert_tile(InsSmem<Q, NW> &S, DevChain *__restrict__ ch,
                                            const int2 *__restrict__ tab, int64_t blk0, int group,
                                            Scratch s) {
  constexpr int WC = InsWarp<NW>::WC;
  // a ticket, or none if the update has stopped: one answer for the block
  if (threadIdx.x == 0) S.gt = halted(s) ? -1 : blk0 + (int64_t)atomicAdd(s.tickets + group, 1u);
  __syncthreads();
  const int64_t gt = S.gt;
  if (gt < 0) return;
  const int2 t = tab[gt];
  DevChain &C = ch[t.x];
  const int cur = C.cur;
  const int32_t *op = C.op_ptr[cur];
  const long long *otau = (const long long *)C.op_tau[cur];
  const uint8_t *s0 = C.s0[cur];
  int32_t *vp = s.vptr + C.cell_off;
  if (threadIdx.x == 0) {
    // Stage the old operator times around the tile with one bulk copy
    // (16-byte bounds: op_tau has room for one time past its capacity),
    // overlapped with the cells' set-up.
    const int R = 8 * Q * Q;
    const int ce = min(C.ncell, t.y * TILE + TILE);
    int lo = op[max(0, t.y * TILE - R)] & ~1, hi = (op[min(C.ncell, ce + R)] + 1) & ~1;
    if (hi - lo > InsStage<Q>::N) {
      lo = op[min(C.ncell, t.y * TILE)] & ~1;
      hi = (op[ce] + 1) & ~1;
      if (hi - lo > InsStage<Q>::N) hi = lo;
    }
    S.slo = lo;
    S.shi = hi;
    mbar_init(&S.bar);
    if (hi > lo) bulk_g2s(S.sop, otau + lo, (uint32_t)(hi - lo) * 8u, &S.bar);
  }
  if (threadIdx.x < KMAX) {
    S.T[0][threadIdx.x] = c_T_full[threadIdx.x];
    S.T[1][threadIdx.x] = C.T_last[threadIdx.x];
  }
  __syncthreads();

  // -- per-cell set-up ---------------------------------------------------------
  const int lane = threadIdx.x & 31, wid = uniform((int)threadIdx.x >> 5), cl = lane & (WC - 1), side = (lane / WC) & 1;
  const int cw = wid * WC + cl, cell = t.y * TILE + cw;
  const bool valid = cell < C.ncell;
  const int slo = S.slo, shi = S.shi;
  // the keys as uniform values: their schedule leaves the vector pipes
  const uint32_t k0 = uniform((uint32_t)C.seed), k1 = uniform((uint32_t)(C.seed >> 32)), sweep = uniform(C.sweep);
  InsCell X{0, 0, 0, 0};
  int q0, q1, par = 0, less = 0;
  bool staged = shi > slo;
  U4 o{0, 0, 0, 0};
  if (valid) {
    cell_bj(C, cell, X.b, X.j);
    o = philox((TAG_INSERT << 24) | (uint32_t)side, (uint32_t)X.b, (uint32_t)X.j, sweep, k0, k1);
    const int u = side ? right_sub<Q>(X.b, C.L) : left_sub<Q>(X.b);
    const int blk = X.j / TW, jb = blk * TW;
    const uint8_t *prow = s.bpar + C.bpar_off + (int64_t)blk * C.nbond;
    int k = side * (2 * Q - 1);
    par = s0[u] & 1;
#pragma unroll
    for (int m = 0; m < 2 * Q; ++m) {
      const int bb = inc_bond<Q>(u, m, C.L);
      if (bb == X.b) continue;
      const int cj = cell_of(C, bb, X.j), cs = cell_of(C, bb, jb);
      const int a = op[cj], e = op[cj + 1];
      par ^= (prow[bb] ^ (a - op[cs])) & 1;
      staged &= a >= slo && e <= shi;
      less |= (bb < X.b ? 1 : 0) << k;
      S.nb[cw][k] = make_int2(a, e);
      ++k;
    }
    q0 = op[cell];
    q1 = op[cell + 1];
    staged &= q0 >= slo && q1 <= shi;
  } else {
    q0 = q1 = op[C.ncell];  // cells past the chain's end: empty ranges
  }
  __syncwarp();
  par ^= __shfl_xor_sync(0xffffffffu, par, WC);
  less |= __shfl_xor_sync(0xffffffffu, less, WC);
  if (valid && !side) {
    S.par0[cw] = (uint8_t)par;
    S.less[cw] = (unsigned short)less;
    S.j[cw] = X.j;
    S.own[cw] = make_int2(q0, q1);
    // K = number of thresholds T[0..KMAX-2] at or below U (they ascend)
    const uint64_t U = (uint64_t)o.x | ((uint64_t)o.y << 32);
    const unsigned long long *T = S.T[X.j == C.nwin - 1 ? 1 : 0];
#pragma unroll
    for (int step = 32; step > 0; step >>= 1)
      if (X.K + step <= KMAX - 1 && T[X.K + step - 1] <= U) X.K += step;
    if ((long long)C.win[3 * X.j + 2] <= 0) X.K = 0;  // empty last window
  }
  __syncwarp();
  X.K = __shfl_sync(0xffffffffu, X.K, cl);
  X.kpre = X.K;
#pragma unroll
  for (int d = 1; d < WC; d <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, X.kpre, d, WC);
    if (cl >= d) X.kpre += y;
  }
  X.kpre -= X.K;
  staged = __all_sync(0xffffffffu, staged || !valid) && shi > slo;
  if (staged && valid && ins_moves<NW>(lane)) {  // ranges from the first staged operator on
    const int n0 = side * (2 * Q - 1);
#pragma unroll
    for (int k = 0; k < 2 * Q - 1; ++k) {
      S.nb[cw][n0 + k].x -= slo;
      S.nb[cw][n0 + k].y -= slo;
    }
    if (!side) S.own[cw] = make_int2(q0 - slo, q1 - slo);
  }
  __syncwarp();
  bool ok = true;
  if (shi > slo) ok = mbar_wait(&S.bar, 0);

  // -- draw, decide, count; then place and write --------------------------------
  const int cap = (C.ins_span >= INS_MIN_SPAN && C.ins_span < InsWarp<NW>::CAP * NW)
                      ? max(KMAX - 1, C.ins_span / NW)
                      : InsWarp<NW>::CAP;
  const bool single = __shfl_sync(0xffffffffu, X.kpre + X.K, WC - 1) <= cap;
  // Vertices of a group of cells: kept candidates placed (marked), all written.
  int nkept = 0, nk = 0, cex = 0;
  auto next = [&](int c0) {  // end of the group that starts at cell c0
    if (single) return WC;
    const int kb = __shfl_sync(0xffffffffu, X.kpre, c0);
    return c0 + __popc(__ballot_sync(0xffffffffu, lane < WC && cl >= c0 && X.kpre + X.K - kb <= cap));
  };
  for (int c0 = 0; c0 < WC;) {
    const int c1 = next(c0);
    nkept = uniform(ins_group<Q, NW>(C, S, otau, wid, X, o, c0, c1, staged, sweep, k0, k1));
    if (cl >= c0 && cl < c1) nk = S.nk[cw];
    c0 = c1;
  }
  const int cnt = q1 - q0 + nk;
  cex = cnt;
#pragma unroll
  for (int d = 1; d < WC; d <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, cex, d, WC);
    if (cl >= d) cex += y;
  }
  if (lane == WC - 1) S.wtot[wid] = cex;
  cex -= cnt;
  if (!__syncthreads_and(ok)) {  // the bulk copy did not arrive within its bound
    if (threadIdx.x == 0) atomicOr(s.status, ST_TIMEOUT);
    return;
  }
  int ctot = 0;
#pragma unroll
  for (int k = 0; k < NW; ++k) {
    if (k == wid) cex += ctot;
    ctot += S.wtot[k];
  }
  // The tile's count goes out before its candidates are placed, the look-back
  // for its offset comes after: by then the tiles before it have mostly
  // published theirs.
  if (threadIdx.x == 0) lb_publish(s.tile_state, gt, t.y == 0 ? LB_INC : LB_AGG, ctot);
  if (lane < WC) S.cex[cw] = cex;
  auto marked = [&](int from, int n) {
    if (n > InsWarp<NW>::MARKS) return false;
    for (int i = lane; i < (n + 3) / 4; i += 32) ((uint32_t *)S.mark[wid])[i] = 0u;
    __syncwarp();
    if (staged)
      ins_place<Q, NW, true, false>(C, S, otau, wid, nkept, from, 0, s);
    else
      ins_place<Q, NW, false, false>(C, S, otau, wid, nkept, from, 0, s);
    return true;
  };
  const int wfrom = __shfl_sync(0xffffffffu, cex, 0), wn = uniform(__shfl_sync(0xffffffffu, cex + cnt, WC - 1) - wfrom);
  __syncwarp();
  bool mk = single && marked(wfrom, wn);
  if (threadIdx.x < 32) {
    int64_t excl = 0;
    if (t.y != 0) {
      excl = lb_lookback(s.tile_state, gt, gt - t.y, s);
      if (threadIdx.x == 0) lb_publish(s.tile_state, gt, LB_INC, excl + ctot);
    }
    if (threadIdx.x == 0) {
      S.excl = excl;
      if (t.y == C.ntile - 1) {
        C.n = excl + ctot;
        if (excl + ctot > C.vcap) atomicOr(s.status, ST_VTX_OVERFLOW);
        // vertex ids are int32 and per-tile loops step past the last id by
        // up to a block: keep every id below 2^31 - 4096
        if (excl + ctot > (int64_t)VTX_ID_LIMIT) atomicOr(s.status, ST_ID_OVERFLOW);
      }
    }
  }
  __syncthreads();
  const int64_t base = S.excl;
  if (base + ctot > C.vcap) return;  // overflow: the host grows the chain and replays
  if (valid && !side) {
    vp[cell] = (int32_t)(base + cex);
    if (cell == C.ncell - 1) vp[C.ncell] = (int32_t)(base + cex + cnt);
  }
  if (!single && valid)  // drawn again group by group
    o = philox((TAG_INSERT << 24) | (uint32_t)side, (uint32_t)X.b, (uint32_t)X.j, sweep, k0, k1);
  for (int c0 = 0; c0 < WC;) {
    const int c1 = next(c0);
    const int qa = __shfl_sync(0xffffffffu, q0, c0), qb = __shfl_sync(0xffffffffu, q1, c1 - 1);
    const int from = __shfl_sync(0xffffffffu, cex, c0), n = uniform(__shfl_sync(0xffffffffu, cex + cnt, c1 - 1) - from);
    if (!single) {
      nkept = ins_group<Q, NW>(C, S, otau, wid, X, o, c0, c1, staged, sweep, k0, k1);
      mk = marked(from, n);
    }
    if (!mk) {
      ins_place<Q, NW, false, true>(C, S, staged ? S.sop : otau, wid, nkept, 0, base, s);
      const int64_t vb = C.vtx_base + base;
      ins_write_old<Q, NW>(S, otau, wid, q0, cex, qa, qb, (long long *)s.vtau + vb, s.vflag + vb, s.vcell + vb);
    } else if (staged) {
      ins_write<Q, NW, true>(C, S, otau, wid, n, from, cex, qa, base, s);
    } else {
      ins_write<Q, NW, false>(C, S, otau, wid, n, from, cex, qa, base, s);
    }
    c0 = c1;
  }
}

// ---- per-chain scan of the tiles' new-operator counts ------------------------------
// A chain's tiles in gridDim.y parts: a part sums its counts, gets the count
// before it by look-back over the parts (all parts of all chains are resident
// at once: see launch_scan_ops), then scans its counts.  One part per chain
// took 0.35 ms of 46 at 2^19 tiles, and 25 us of 3 ms at 2^15.
__global__ void __launch_bounds__(1024) k_scan_ops(DevChain *__restrict__ ch, Scratch s) {
  // Chunks of 4 x 1024 tiles: each thread loads four consecutive counts
  // (coalesced across the warp), one block scan per chunk; the next chunk's
  // loads are issued before the current chunk's scan.
  __shared__ int64_t sm[33];
  __shared__ int64_t before;
  if (halted_block(s)) return;
  DevChain &C = ch[blockIdx.x];
  const int per = (C.ntile + gridDim.y - 1) / gridDim.y;
  const int i0 = min(C.ntile, (int)blockIdx.y * per), nt = min(C.ntile, i0 + per) - i0;
  const int64_t *cnt = s.tile_sum2 + C.tile0 + i0;
  int64_t *pref = s.tile_pref2 + C.tile0 + i0;
  constexpr int V = 4;
  const int chunk = V * (int)blockDim.x;
  int64_t v[V], nx[V];
  auto load = [&](int base, int64_t *x) {
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const int i = base + V * (int)threadIdx.x + k;
      x[k] = (i < nt) ? cnt[i] : 0;
    }
  };
  int64_t run = 0;
  if (gridDim.y > 1) {
    int64_t mine = 0;
    for (int i = threadIdx.x; i < nt; i += blockDim.x) mine += cnt[i];
    const int64_t sum = block_sum<int64_t>(mine, sm);
    if (threadIdx.x < 32) {
      const int64_t p0 = (int64_t)blockIdx.x * gridDim.y, p = p0 + blockIdx.y;
      int64_t excl = 0;
      if (blockIdx.y) {
        if (threadIdx.x == 0) lb_publish(s.part_state, p, LB_AGG, sum);
        __syncwarp();
        excl = lb_lookback(s.part_state, p, p0, s);
      }
      if (threadIdx.x == 0) {
        lb_publish(s.part_state, p, LB_INC, excl + sum);
        before = excl;
      }
    }
    __syncthreads();
    run = before;
  }
  load(0, v);
  for (int base = 0; base < nt; base += chunk) {
    if (base + chunk < nt) load(base + chunk, nx);
    int64_t mine = 0;
#pragma unroll
    for (int k = 0; k < V; ++k) mine += v[k];
    int64_t total;
    int64_t ex = run + block_excl_scan<int64_t>(mine, sm, total);
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const int i = base + V * (int)threadIdx.x + k;
      if (i < nt) pref[i] = ex;
      ex += v[k];
    }
    run += total;
#pragma unroll
    for (int k = 0; k < V; ++k) v[k] = nx[k];
  }
  if (threadIdx.x == 0 && blockIdx.y == gridDim.y - 1) {
    C.n_off_new = run;
    if (run > C.op_cap) atomicOr(s.status, ST_OP_OVERFLOW);
  }
}

// ---- tau = 0: last leg per subsite, subspin permutation, cut predecessors -----
// One thread per subsite: the last vertex on its 2 Q bonds.  The bonds' last
// windows are read side by side (a thread per site that walked them one after
// another took 22 us at S = 2, one dependent load after the other); only a bond
// whose last window is empty is walked further down.
template <int Q>
__global__ void __launch_bounds__(SITE_BLOCK * Q) k_cut(const DevChain *__restrict__ ch,
                                                    const int2 *__restrict__ tab, int64_t blk0,
                                                    Scratch s) {
  __shared__ int slast[SITE_BLOCK * Q];
  __shared__ uint8_t stop_[SITE_BLOCK * Q];
  if (halted_block(s)) return;
  const int2 t = tab[blk0 + blockIdx.x];
  const DevChain &C = ch[t.x];
  const int u = t.y * SITE_BLOCK * Q + threadIdx.x, i = u / Q;  // subsite, site
  const int32_t *vp = s.vptr + C.cell_off;
  const long long *vt = (const long long *)s.vtau + C.vtx_base;
  const uint8_t *s0 = C.s0[C.cur];
  const uint8_t *ptot = s.bpar + C.bpar_off + (int64_t)C.nblk * C.nbond;
  if (i < C.L) {
    int best = -1, par = 0;
    long long bt = 0;
    int id[2 * Q];
#pragma unroll
    for (int m = 0; m < 2 * Q; ++m) {
      const int bb = inc_bond<Q>(u, m, C.L);
      par ^= ptot[bb];
      const int c = cell_of(C, bb, C.nwin - 1);
      const int a = vp[c], e = vp[c + 1];
      id[m] = e > a ? e - 1 : -1;
    }
#pragma unroll
    for (int m = 0; m < 2 * Q; ++m) {
      if (id[m] >= 0) continue;
      const int bb = inc_bond<Q>(u, m, C.L);
      for (int j = C.nwin - 2; j >= 0; --j) {
        const int c = cell_of(C, bb, j);
        const int a = vp[c], e = vp[c + 1];
        if (e > a) {
          id[m] = e - 1;
          break;
        }
      }
    }
    long long tt[2 * Q];
#pragma unroll
    for (int m = 0; m < 2 * Q; ++m) tt[m] = id[m] >= 0 ? vt[id[m]] : 0;
#pragma unroll
    for (int m = 0; m < 2 * Q; ++m)
      if (id[m] >= 0 && (best < 0 || tt[m] > bt || (tt[m] == bt && id[m] > best))) {
        best = id[m];
        bt = tt[m];
      }
    slast[threadIdx.x] = best;
    stop_[threadIdx.x] = (uint8_t)((s0[u] ^ par) & 1);
  }
  __syncthreads();
  if (i >= C.L) return;
  // Every subsite's thread takes its site's permutation (the same on all of them).
  int last[Q], top[Q];
  const int k0 = (int)threadIdx.x / Q * Q;  // the site's first thread
#pragma unroll
  for (int a = 0; a < Q; ++a) {
    last[a] = slast[k0 + a];
    top[a] = stop_[k0 + a];
  }
  // perm[a]: the bottom subspin that the top of subspin a continues into.
  int perm[Q];
  if (Q == 1) {
    perm[0] = 0;
  } else if (Q > 2) {
    // Uniform among the permutations that join every top to a bottom of the
    // same spin (heat bath of the symmetrization, Sec. 5): tops and bottoms of
    // spin 1, then of spin 0, in subspin order; each bottom list shuffled by
    // Fisher-Yates from the last place down, place j drawn as
    // floor(w (j+1) / 2^32) with w the next word of
    // Philox(((TAG_PERM << 24) | 1, i, 0, sweep)); the m-th top of each spin
    // continues into the m-th shuffled bottom.
    int tops[2][Q], bots[2][Q], nt[2] = {0, 0}, nb[2] = {0, 0};
#pragma unroll
    for (int a = 0; a < Q; ++a) {
      const int gt = top[a] ? 0 : 1, gb = (s0[i * Q + a] & 1) ? 0 : 1;
      tops[gt][nt[gt]++] = a;
      bots[gb][nb[gb]++] = a;
    }
#pragma unroll
    for (int a = 0; a < Q; ++a) perm[a] = a;
    if (nt[0] != nb[0]) {
      atomicOr(s.status, ST_BADSTATE);
    } else {
      const U4 o = philox((TAG_PERM << 24) | 1u, (uint32_t)i, 0u, C.sweep, (uint32_t)C.seed,
                          (uint32_t)(C.seed >> 32));
      const uint32_t w[4] = {o.x, o.y, o.z, o.w};
      int d = 0;
      for (int g = 0; g < 2; ++g) {
        for (int j = nb[g] - 1; j >= 1; --j) {
          const int r = (int)__umulhi(w[d++ & 3], (uint32_t)(j + 1));
          const int tmp = bots[g][j];
          bots[g][j] = bots[g][r];
          bots[g][r] = tmp;
        }
        for (int m = 0; m < nt[g]; ++m) perm[tops[g][m]] = bots[g][m];
      }
    }
  } else {
    const int b0 = s0[i * Q] & 1, b1 = s0[i * Q + (Q > 1 ? 1 : 0)] & 1;
    const bool ok_id = (top[0] == b0) && (top[1] == b1);
    const bool ok_sw = (top[0] == b1) && (top[1] == b0);
    int sw;
    if (ok_id && ok_sw)
      sw = coin(C, TAG_PERM, (uint32_t)i);
    else if (ok_sw)
      sw = 1;
    else if (ok_id)
      sw = 0;
    else {
      atomicOr(s.status, ST_BADSTATE);
      sw = 0;
    }
    perm[0] = sw ? 1 : 0;
    perm[1] = sw ? 0 : 1;
  }
  // Walk down through the cut: the bottom of subspin a is entered from the
  // top of pinv(a), then possibly through empty subspins.
  const int a = u - i * Q;
  int x = a, cross = 0, node = -1, mn = a, len = 0;
  for (int step = 0; step < Q; ++step) {
    int y = 0;
#pragma unroll
    for (int z = 0; z < Q; ++z)
      if (perm[z] == x) y = z;
    x = y;
    ++cross;
    int lx = 0;
#pragma unroll
    for (int z = 0; z < Q; ++z)
      if (z == x) lx = last[z];
    if (lx >= 0) {
      node = lx;
      break;
    }
    mn = min(mn, x);
    ++len;
    if (x == a) break;
  }
  const int64_t v = C.sub_off + u;
  s.cut_node[v] = node;
  s.cut_cross[v] = (int8_t)cross;
  s.free_min[v] = (node < 0) ? i * Q + mn : -1;
  s.free_len[v] = (int8_t)len;
}

// ---- linking + union-find -----------------------------------------------------
__device__ __forceinline__ int before_window(const DevChain &C, const int32_t *vp, int bond, int j) {
  for (int jj = j - 1; jj >= 0; --jj) {
    const int c = cell_of(C, bond, jj);
    const int a = vp[c], e = vp[c + 1];
    if (e > a) return e - 1;
  }
  return -1;
}

// Per-cell linking context, staged in shared memory by one thread per cell.
template <int Q>
struct LinkCell {
  static constexpr int NO = 2 * Q - 1;  // other bonds touching each of the two subsites
  int wa[2][NO], we[2][NO], bj[2][NO];
  int own_bj, cut[2];
};

// Union-find of one tile's nodes in shared memory (local ids), with the same
// min-root rule as the global one: lp[x] <= x; a link is one CAS on the larger
// root.  Walks are bounded by the tile's node count.
__device__ __forceinline__ int suf_find(volatile int *lp, int x, int bound, int *status) {
  for (int it = 0; it <= bound; ++it) {
    const int p = lp[x];
    if (p == x) return x;
    const int g = lp[p];
    if (g != p) lp[x] = g;  // path halving (g is an ancestor of x)
    x = g;
  }
  atomicOr(status, ST_TIMEOUT);
  return x;
}

__device__ __forceinline__ void suf_union(int *lp, int a, int b, int bound, int *status) {
  for (int it = 0; it <= bound; ++it) {
    a = suf_find(lp, a, bound, status);
    b = suf_find(lp, b, bound, status);
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

// First index q in [lo, hi) with vt[q] >= thr.  For a neighbour cell, whose
// ids are all below w or all above it, "key (tau, id) below (tw, w)" is
// vt[q] < tw + 1 or vt[q] < tw respectively.  A cell holds 11 vertices on
// average: more than 15 are halved first, then four steps without branches,
// each reading up to VTX_PAD - 1 times past hi.
__device__ __forceinline__ int time_lower_bound(const long long *vt, int lo, int hi, long long thr) {
  while (hi - lo > 15) {
    const int mid = lo + ((hi - lo) >> 1);  // no overflow near 2^31
    if (vt[mid] < thr)
      lo = mid + 1;
    else
      hi = mid;
  }
  int rem = hi - lo;
  const long long *p = vt + lo;
#pragma unroll
  for (int d = 8; d > 0; d >>= 1) {
    const bool in = rem >= d, below = p[d - 1] < thr;
    const int go = (in & below) ? d : 0;
    p += go;
    rem -= go;
  }
  return hi - rem;
}

// Linking, then the union of the two fragments below every vertex.  Edges
// with both nodes in the tile are united in shared memory, and the tile's
// forest is then stored flat: every node points at its tile component's
// root, its smallest node.  Edges
// that leave the tile are marked and united in the global forest by k_link_x,
// after every tile has stored its forest (a tile too large for shared memory
// leaves all of its edges to k_link_x, with every node its own root).
template <int Q, int NT>
__global__ void __launch_bounds__(NT, 2048 / NT) k_link(const DevChain *__restrict__ ch,
                                              const int2 *__restrict__ tab, int64_t blk0,
                                              Scratch s) {
  __shared__ LinkCell<Q> lc[TILE];
  __shared__ int cvp[TILE + 1];
  __shared__ int lp[SMEM_CAP];
  __shared__ uint32_t equeue[NT / 32][64];  // per warp: edges to unite
  __shared__ int stop;
  if (threadIdx.x == 0) stop = halted(s);
  const int2 t = tab[blk0 + blockIdx.x];
  const DevChain &C = ch[t.x];
  const int c0 = t.y * TILE, c1 = min(C.ncell, c0 + TILE), ncl = c1 - c0;
  const int32_t *vp = s.vptr + C.cell_off;
  for (int i = threadIdx.x; i <= ncl; i += blockDim.x) cvp[i] = vp[c0 + i];
  if (threadIdx.x < ncl) {
    LinkCell<Q> &L = lc[threadIdx.x];
    int b, j;
    cell_bj(C, c0 + threadIdx.x, b, j);
    const int sub[2] = {left_sub<Q>(b), right_sub<Q>(b, C.L)};
#pragma unroll
    for (int sd = 0; sd < 2; ++sd) {
      int k = 0;
#pragma unroll
      for (int m = 0; m < 2 * Q; ++m) {
        const int bb = inc_bond<Q>(sub[sd], m, C.L);
        if (bb == b) continue;
        const int cj = cell_of(C, bb, j);
        L.wa[sd][k] = vp[cj];
        L.we[sd][k] = vp[cj + 1];
        L.bj[sd][k] = before_window(C, vp, bb, j);
        ++k;
      }
      L.cut[sd] = s.cut_node[C.sub_off + sub[sd]];
    }
    L.own_bj = before_window(C, vp, b, j);
  }
  __syncthreads();
  if (stop) return;
  const int a = cvp[0], e = cvp[ncl], nv = e - a;
  const bool local = nv <= local_cap(C);
  if (local)
    for (int i = threadIdx.x; i < nv; i += blockDim.x) lp[i] = i;
  __syncthreads();
  const int64_t vb = C.vtx_base, wb = vb >> 5;
  const long long *__restrict__ vt = (const long long *)s.vtau + vb;
  int32_t *par = s.parent + vb;
  // Whole warps walk the tile (trip count rounded up).  About half of the
  // vertices have an edge to unite in the tile.  Most find their larger node
  // still its own parent: one compare-and-swap hangs it below the smaller one
  // without looking for roots.  Else the node's parent and the smaller node are to
  // be united; a warp queues these and unites 32 at a time with all lanes.  At
  // L=16384, beta=4096: 0.607 -> 0.575 ms against queueing every edge (S=1, L=4096:
  // 0.265 -> 0.255), 0.675 -> 0.638 queueing against uniting each step's edges (both
  // with k_link_x); a second such try before queueing gains nothing.
  const int lane = threadIdx.x & 31;
  uint32_t *queue = equeue[threadIdx.x >> 5];
  int nqueue = 0;
  for (int w0 = a + (int)(threadIdx.x & ~31u); w0 < e; w0 += blockDim.x) {
    const int w = w0 + lane;
    uint32_t edge = 0u;  // the two nodes' indices in the tile; 0: none (they differ)
    if (w < e) {
      const int ci = s.vcell[vb + w];
      const LinkCell<Q> &L = lc[ci];
      const long long tw = vt[w];
      const int own = w > cvp[ci] ? w - 1 : L.own_bj;  // on the vertex's own bond
      const long long ot = own >= 0 ? vt[own] : 0;
      int P[2];
      uint8_t wrapbits = 0;
#pragma unroll
      for (int sd = 0; sd < 2; ++sd) {
        int best = own;
        long long bt = ot;
#pragma unroll
        for (int k = 0; k < LinkCell<Q>::NO; ++k) {
          const int q = time_lower_bound(vt, L.wa[sd][k], L.we[sd][k], tw + (L.wa[sd][k] < w ? 1 : 0));
          const int cand = (q > L.wa[sd][k]) ? q - 1 : L.bj[sd][k];
          if (cand >= 0) {
            const long long tc = vt[cand];
            if (best < 0 || tc > bt || (tc == bt && cand > best)) {
              best = cand;
              bt = tc;
            }
          }
        }
        if (best < 0) {
          best = L.cut[sd];
          wrapbits |= sd ? VF_WRAP_R : VF_WRAP_L;
          if (best < 0) {
            fail_check(s, 2, c0 + ci, w, sd, 0, 0);
            best = w;
          }
        }
        P[sd] = best;
      }
      s.pl[vb + w] = P[0];
      s.pr[vb + w] = P[1];
      if (wrapbits) s.vflag[vb + w] |= wrapbits;
      const bool inside = P[0] >= a && P[0] < e && P[1] >= a && P[1] < e;
      if (!inside) {
        set_bit(s.openmark, wb, P[0]);
        if (local && P[0] != P[1]) set_bit(s.xmark, wb, w);
      } else if (local && P[0] != P[1]) {
        const int lo = min(P[0], P[1]) - a, hi = max(P[0], P[1]) - a;
        const int old = atomicCAS(lp + hi, hi, lo);
        if (old != hi && old != lo) edge = (uint32_t)lo | ((uint32_t)old << 16);
      }
    }
    const unsigned m = __ballot_sync(0xffffffffu, edge != 0u);
    if (edge) queue[nqueue + __popc(m & ((1u << lane) - 1u))] = edge;
    nqueue += __popc(m);
    __syncwarp();
    if (nqueue >= 32) {
      nqueue -= 32;
      const uint32_t x = queue[nqueue + lane];
      suf_union(lp, x & 0xffffu, x >> 16, nv, s.status);
      __syncwarp();
    }
  }
  if (lane < nqueue) {
    const uint32_t x = queue[lane];
    suf_union(lp, x & 0xffffu, x >> 16, nv, s.status);
  }
  __syncthreads();
  if (local) {
    // Every node walks to its root and stores it (in shared memory too, which
    // shortens the walks of the nodes below it).  Each store writes an
    // ancestor of the old word, so concurrent walks still end at the root;
    // the walks are bounded by the tile's node count.  One pass without
    // barriers (pointer jumping, one barrier per round: 0.83 -> 0.81 ms at
    // L=16384, beta=4096).
    volatile int *vlp = lp;
    for (int i = threadIdx.x; i < nv; i += blockDim.x) {
      int r = vlp[i];
      for (int it = 0; it < SMEM_CAP; ++it) {
        const int q = vlp[r];
        if (q == r) break;
        r = q;
      }
      vlp[i] = r;
      par[a + i] = a + r;
    }
  } else {
    for (int v = a + threadIdx.x; v < e; v += blockDim.x) par[v] = v;
  }
}

// Union that tries one compare-and-swap on the nodes' parents (tile roots) before
// it looks for global roots: L=16384, beta=4096 linking + unions 0.688 -> 0.679 ms,
// S=1, L=4096 0.312 -> 0.305 (no difference in k_link_xt, whose time is the
// longest chain).
__device__ __forceinline__ void uf_union_try(int32_t *par, int a, int b, int *status, int limit) {
  const int ra = __ldcg(par + a), rb = __ldcg(par + b);
  if (ra == rb) return;
  const int lo = min(ra, rb), hi = max(ra, rb);
  const int old = atomicCAS(par + hi, hi, lo);
  if (old != hi && old != lo) uf_union(par, lo, old, status, limit);
}

// Global unions of the edges that leave their tile (all edges of a tile too
// large for shared memory), on the forests the tiles stored.  One warp per
// tile, eight tiles per block: a tile has about 45 words of marks, and the
// unions are chains of dependent global loads, so many tiles are kept in
// flight.
constexpr int TPB_X = 256;
constexpr int XLIST = 256;  // crossing edges of a tile listed per warp

__global__ void __launch_bounds__(TPB_X) k_link_x(const DevChain *__restrict__ ch,
                                                const int2 *__restrict__ tab, int64_t ntiles,
                                                Scratch s) {
  __shared__ int xlist[TPB_X / 32][XLIST];
  if (halted_warp(s)) return;
  const int lane = threadIdx.x & 31;
  const int64_t gt = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (gt >= ntiles) return;
  const int2 t = tab[gt];
  const DevChain &C = ch[t.x];
  const int c0 = t.y * TILE, c1 = min(C.ncell, c0 + TILE);
  const int32_t *vp = s.vptr + C.cell_off;
  const int a = vp[c0], e = vp[c1];
  const bool local = e - a <= local_cap(C);
  const int64_t vb = C.vtx_base;
  int32_t *par = s.parent + vb;
  if (!local) {
    for (int w = a + lane; w < e; w += 32) uf_union(par, s.pl[vb + w], s.pr[vb + w], s.status, s.uf_limit);
    return;
  }
  // The tile's crossing edges cluster at its first vertices (its first bond's
  // cells): they are listed first (a warp scan of the mark words' counts) and
  // then taken round-robin by the lanes, so that no lane walks most of them.
  int *list = xlist[threadIdx.x >> 5];
  const int64_t wfirst = (vb + a) >> 5, wlast = (vb + e - 1) >> 5;
  int nlist = 0;
  for (int64_t w0 = wfirst; e > a && w0 <= wlast; w0 += 32) {  // the same trip count on every lane
    const int64_t wd = w0 + lane;
    uint32_t bits = 0u;
    const int64_t v0 = (wd << 5) - vb;
    if (wd <= wlast) {
      bits = __ldcg(s.xmark + wd);
      if (v0 < a) bits &= ~0u << (a - v0);
      if (v0 + 32 > e) bits &= (e - v0 >= 32) ? ~0u : ((1u << (e - v0)) - 1u);
    }
    const int cnt = __popc(bits);
    int inc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    int at = nlist + inc - cnt;
    while (bits) {
      const int w = (int)v0 + __ffs(bits) - 1;
      bits &= bits - 1;
      if (at < XLIST)
        list[at] = w;
      else
        uf_union(par, s.pl[vb + w], s.pr[vb + w], s.status, s.uf_limit);  // past the list
      ++at;
    }
    nlist += __shfl_sync(0xffffffffu, inc, 31);
  }
  __syncwarp();
  for (int i = lane; i < min(nlist, XLIST); i += 32) {
    const int w = list[i];
    uf_union_try(par, s.pl[vb + w], s.pr[vb + w], s.status, s.uf_limit);
  }
}

// The same unions with one block per tile, for launches of few tiles: there
// the time is the chain of dependent L2 accesses of the slowest warp, not the
// work.  The block lists the tile's crossing edges (a warp takes a mark word at
// a time, one bit per lane; S >= 1 tiles have hundreds, 300 to 700 of 1000
// edges), every thread unites edges of the list and then walks once more from
// one node of each of its edges: the walks of all threads halve the same long
// paths (min-root links chain the tiles of a loop), so that the waiting unions
// and the compression find short ones.  linking + unions / compression, us:
// S = 2, 65 tiles 213 / 32 -> 90 / 23; S = 3/2, 1024 tiles 244 / 46 -> 122 /
// 37; S = 1/2, 128 tiles 47 / 28 -> 40 / 20.  Without the second walk the
// unions got faster but the compression slower (S = 2: 108 / 49).
// Up to how many tiles per launch: where a warp per tile becomes as fast.  One
// update in us, block / warp per tile: S = 1/2, 64 tiles 71.7 / 75.2, 512 122 / 128,
// 1024 173 / 179, 1280 206 / 208, 1408 217 / 217, 2048 258 / 257, 3000 344 / 342
// (beta = 4, loops that span few tiles: 2048 140 / 136, 3072 180 / 175); S = 1, 512
// 140 / 151, 1024 190 / 199, 2048 305 / 306, 3000 411 / 407; S = 2,
// beta = 512: 2048 595 / 662, 3040 793 / 828, 3600 889 / 903, 4096 1026 / 1021.  S = 3/2
// has S = 2's line, which is on the safe side of its own (3040 609 / 704, 4096 766 / 838,
// 6000 1041 / 1084).
constexpr int64_t xt_max_tiles(int Q) { return 152 * (Q == 1 ? 8 : Q == 2 ? 12 : 20); }

__global__ void __launch_bounds__(TPB_X) k_link_xt(const DevChain *__restrict__ ch,
                                                const int2 *__restrict__ tab, int64_t blk0,
                                                Scratch s) {
  __shared__ unsigned short xlist[SMEM_CAP];
  __shared__ int nx;
  __shared__ int stop;
  if (threadIdx.x == 0) stop = halted(s);
  const int2 t = tab[blk0 + blockIdx.x];
  const DevChain &C = ch[t.x];
  const int c0 = t.y * TILE, c1 = min(C.ncell, c0 + TILE);
  const int32_t *vp = s.vptr + C.cell_off;
  const int a = vp[c0], e = vp[c1];
  const int64_t vb = C.vtx_base;
  int32_t *par = s.parent + vb;
  if (threadIdx.x == 0) nx = 0;
  __syncthreads();
  if (stop) return;
  if (e - a > local_cap(C)) {  // every edge of the tile
    for (int w = a + threadIdx.x; w < e; w += TPB_X)
      uf_union(par, s.pl[vb + w], s.pr[vb + w], s.status, s.uf_limit);
    return;
  }
  constexpr int NW = TPB_X / 32;
  constexpr int WMAX = (SMEM_CAP / 32 + 1 + NW - 1) / NW;  // mark words per warp
  static_assert(WMAX <= 32, "one lane loads each mark word of a warp");
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t wfirst = (vb + a) >> 5, wlast = (vb + e - 1) >> 5;
  uint32_t mine = 0u;
  {
    const int64_t wd = wfirst + wid + NW * lane;
    if (lane < WMAX && e > a && wd <= wlast) {
      const int64_t v0 = (wd << 5) - vb;
      mine = __ldcg(s.xmark + wd);
      if (v0 < a) mine &= ~0u << (a - v0);
      if (v0 + 32 > e) mine &= (e - v0 >= 32) ? ~0u : ((1u << (e - v0)) - 1u);
    }
  }
  for (int k = 0; k < WMAX; ++k) {
    const uint32_t bits = __shfl_sync(0xffffffffu, mine, k);
    if (!bits) continue;
    int at = 0;
    if (lane == 0) at = atomicAdd(&nx, __popc(bits));
    at = __shfl_sync(0xffffffffu, at, 0) + __popc(bits & ((1u << lane) - 1u));
    if ((bits >> lane) & 1u)
      xlist[at] = (unsigned short)(((wfirst + wid + NW * k) << 5) + lane - vb - a);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nx; i += TPB_X) {
    const int64_t w = vb + a + xlist[i];
    uf_union(par, s.pl[w], s.pr[w], s.status, s.uf_limit);
  }
  for (int i = threadIdx.x; i < nx; i += TPB_X) {
    const int p = s.pl[vb + a + xlist[i]];
    const int r = uf_find(par, p, s.status, s.uf_limit);
    if (r != p) par[p] = r;  // an ancestor, as in the walk itself
  }
}

// ---- compression + coins --------------------------------------------------------
// Every node's root, and the flip of its loop (one coin per root) as one bit
// per node: the later kernels read flips by node, without the root.
//
// Only this block writes parent words of [a, e) in this kernel, and every word
// it writes is an ancestor of the old one: the tile's copy stays a valid forest.
// Words that point out of the tile (parents are never larger than their
// children, so outside means below a) are resolved first, each with one global
// walk to its root and that root's coin, so that the nodes walking through
// them share both; every other walk then stays in shared memory.  In the
// tile's copy a word is the parent's index in the tile, or, with the top bit
// set, the root outside.  The shared copy and the global words agree after
// that pass, and a node's word is stored only if its root differs from it
// (linking left most words at their root: 0.31 -> 0.28 ms at L=16384,
// beta=4096).
constexpr unsigned OUTSIDE = 0x80000000u;
constexpr int COIN_GROUPS = SMEM_CAP / 128 + 2;  // Philox blocks of 128 coins a tile in shared memory spans

template <int NT>
__global__ void __launch_bounds__(NT, 2048 / NT) k_compress(const DevChain *__restrict__ ch,
                                                   const int2 *__restrict__ tab, int64_t blk0,
                                                   Scratch s) {
  __shared__ U4 coins[COIN_GROUPS];
  __shared__ int64_t sm[33];
  __shared__ unsigned spar[SMEM_CAP];
  __shared__ uint32_t ocoin[SMEM_CAP / 32 + 2];  // coins of the outside roots, at the nodes that point there
  __shared__ unsigned short olist[SMEM_CAP];     // those nodes
  __shared__ int nout;
  __shared__ int stop;
  if (threadIdx.x == 0) stop = halted(s);
  const int64_t gt = blk0 + blockIdx.x;
  const int2 t = tab[gt];
  const DevChain &C = ch[t.x];
  const int c0 = t.y * TILE, c1 = min(C.ncell, c0 + TILE);
  const int32_t *vp = s.vptr + C.cell_off;
  const int a = uniform(vp[c0]), e = uniform(vp[c1]);
  const int64_t vb = C.vtx_base, wb = vb >> 5;
  int32_t *par = s.parent + vb;
  // (unsigned: a stopped update's offsets may be anything, and give no more groups
  // of coins than there is room for)
  const bool oversized = (unsigned)e - (unsigned)a > (unsigned)local_cap(C);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int step = blockDim.x, first = (a & ~31) + 32 * wid;  // words of 32 vertices, a warp each
  const int g0 = a >> 7;
  const int ng = (e > a && !oversized) ? ((e - 1) >> 7) - g0 + 1 : 0;
  const uint32_t k0 = uniform((uint32_t)C.seed), k1 = uniform((uint32_t)(C.seed >> 32)), sweep = uniform(C.sweep);
  for (int g = threadIdx.x; g < ng; g += blockDim.x)
    coins[g] = philox(TAG_FLIP << 24, (uint32_t)(g0 + g), 0u, sweep, k0, k1);
  if (threadIdx.x == 0) nout = 0;
  for (int i = threadIdx.x; i < SMEM_CAP / 32 + 2; i += blockDim.x) ocoin[i] = 0u;
  __syncthreads();
  if (stop) return;
  if (!oversized) {
    for (int v0 = first; v0 < e; v0 += step) {
      const int v = v0 + lane;
      const bool in = v >= a && v < e;
      const int p = in ? __ldcg(par + v) : a;
      const unsigned m = __ballot_sync(0xffffffffu, p < a);
      if (m) {  // about 5 % of the nodes: listed, so that whole warps take them below
        int at = 0;
        if (lane == 0) at = atomicAdd(&nout, __popc(m));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (p < a) olist[at + __popc(m & ((1u << lane) - 1u))] = (unsigned short)(v - a);
      }
      if (in) spar[v - a] = p < a ? (OUTSIDE | (unsigned)p) : (unsigned)(p - a);
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < nout; k += blockDim.x) {
    const int i = olist[k], v = a + i, p = (int)(spar[i] & ~OUTSIDE);
    const int q = uf_root(par, p, s.status, s.uf_limit);
    if (q != p) {
      par[v] = q;
      spar[i] = OUTSIDE | (unsigned)q;
    }
    if (coin_from(philox(TAG_FLIP << 24, (uint32_t)q >> 7, 0u, sweep, k0, k1), (uint32_t)q))
      atomicOr(&ocoin[(v >> 5) - (a >> 5)], 1u << (v & 31));
  }
  __syncthreads();
  const uint32_t *cw = (const uint32_t *)coins;
  int64_t roots = 0;
  for (int v0 = first; v0 < e; v0 += step) {
    const int v = v0 + lane;
    const bool in = v >= a && v < e;
    int r = -1, flip = 0;
    if (in && !oversized) {
      // the walk ends at a root of the tile, or at a word that points outside
      const unsigned x0 = spar[v - a];
      unsigned k = (unsigned)(v - a), x = x0;
      for (int it = 0; x != k && !(x & OUTSIDE) && it < SMEM_CAP; ++it) {
        k = x;
        x = spar[k];
      }
      if (x & OUTSIDE) {
        r = (int)(x & ~OUTSIDE);
        const int y = a + (int)k;
        flip = (ocoin[(y >> 5) - (a >> 5)] >> (y & 31)) & 1;
        if (x0 != x) par[v] = r;
      } else {
        r = a + (int)k;
        flip = (int)((cw[(r >> 5) - (g0 << 2)] >> (r & 31)) & 1u);
        if (x0 != k) par[v] = r;
      }
    } else if (in) {
      r = uf_root(par, v, s.status, s.uf_limit);
      if (r != v) par[v] = r;
      flip = coin_from(philox(TAG_FLIP << 24, (uint32_t)r >> 7, 0u, sweep, k0, k1), (uint32_t)r);
    }
    const unsigned fm = __ballot_sync(0xffffffffu, flip), rm = __ballot_sync(0xffffffffu, in && r == v);
    if (lane == 0) {
      roots += __popc(rm);
      store_word(s.flipbits, wb + (v0 >> 5), fm, v0, a, e);
      if (oversized && rm) atomicOr(s.openroot + wb + (v0 >> 5), rm);
    }
    const uint32_t om = __ldcg(s.openmark + wb + (v0 >> 5));
    if (in && ((om >> lane) & 1u)) set_bit(s.openroot, wb, r);
  }
  const int64_t tot = block_sum<int64_t>(roots, sm);
  if (threadIdx.x == 0) s.tile_roots[gt] = tot;
}

// ---- opt-in check of the loop forest after compression ----------------------------
// Every node's word is its loop's root, a root is its own parent and no parent
// is larger than its child (min-root rule).  The first violation is reported
// as consistency check 10 (chain, node, word, word of the word).
__global__ void __launch_bounds__(TILE) k_check_forest(const DevChain *__restrict__ ch,
                                                       const int2 *__restrict__ tab, Scratch s) {
  if (halted(s)) return;
  const int2 t = tab[blockIdx.x];
  const DevChain &C = ch[t.x];
  const int c0 = t.y * TILE, c1 = min(C.ncell, c0 + TILE);
  const int32_t *vp = s.vptr + C.cell_off;
  const int a = vp[c0], e = vp[c1];
  const int32_t *par = s.parent + C.vtx_base;
  for (int v = a + threadIdx.x; v < e; v += blockDim.x) {
    const int r = __ldcg(par + v);
    const int rr = (r >= 0 && r <= v) ? __ldcg(par + r) : -1;
    if (r < 0 || r > v || rr != r) fail_check(s, 10, t.x, v, r, rr, 0);
  }
}

// ---- loop properties, new flags ---------------------------------------------------
// Exact 64-bit two's-complement sums kept in shared memory as two 32-bit words
// and added with native 32-bit atomics (a 64-bit shared-memory add would be a
// compare-and-swap loop): the low word first, then the high word plus the
// carry out of the low word.
__device__ __forceinline__ void sadd64(unsigned *w, long long x) {
  const unsigned lo = (unsigned)x, hi = (unsigned)((unsigned long long)x >> 32);
  const unsigned old = atomicAdd(w, lo);
  const unsigned h = hi + ((old + lo < old) ? 1u : 0u);
  if (h) atomicAdd(w + 1, h);
}

__device__ __forceinline__ unsigned long long sget64(const unsigned *w) {
  return ((unsigned long long)w[1] << 32) | w[0];
}

// Per-tile table of loop sums keyed by root: a vertex of a loop of more than
// one node adds its (W, C, S, Zr, Zi) to its root's slot (linear probing,
// split sums).  If the table is full the sums go to the root's global record
// and the root is marked open, so that they are squared with the open loops.
constexpr int LOOP_SLOTS = 256;
constexpr int LOOP_SUMS = 5;  // W, C, S, Zr, Zi

struct LoopSums {
  long long v[LOOP_SUMS];
};

// Adds a loop's first NS sums to the global record of its root (vertex v):
// W, C, S, Zr in one 32-byte record, Zi beside it in its own array.
template <int NS>
__device__ __forceinline__ void acc_add(const Scratch &s, int64_t v, const long long *x) {
  unsigned long long *r = s.acc + ACC_WORDS * v;
#pragma unroll
  for (int i = 0; i < NS; ++i) atomicAdd(i < ACC_WORDS ? r + i : s.accz + v, (unsigned long long)x[i]);
}

// NS: how many of the sums are carried (3 without the temporal moment).
// mask = slots in use - 1 (LOOP_SLOTS - 1 unless a test shrinks the table).
template <int NS>
__device__ __forceinline__ void loop_add(int *keys, unsigned *vals, int key, const LoopSums &x,
                                         const Scratch &s, int64_t vb, unsigned mask) {
  unsigned h = (((unsigned)key * 2654435761u) >> 24) & mask;  // top 8 bits: LOOP_SLOTS = 256
  for (unsigned probe = 0; probe <= mask; ++probe) {
    int k = keys[h];
    if (k == -1) {
      k = atomicCAS(keys + h, -1, key);
      if (k == -1) k = key;
    }
    if (k == key) {
#pragma unroll
      for (int i = 0; i < NS; ++i) sadd64(vals + 2 * (NS * h + i), x.v[i]);
      return;
    }
    h = (h + 1) & mask;
  }
  acc_add<NS>(s, vb + key, x.v);
  set_bit(s.openroot, vb >> 5, key);
}

// A 128-bit sum in four 32-bit words, and the square of |v| < 2^62 added to it:
// ten multiply-adds with carry (the compiler's 64 x 64 -> 128-bit product and
// 128-bit add took about twice that).
struct Sum128 {
  uint32_t a = 0, b = 0, c = 0, d = 0;
  __device__ __forceinline__ void add_square(long long v) {
    const unsigned long long m = (unsigned long long)(v < 0 ? -v : v);
    const uint32_t lo = (uint32_t)m, hi = (uint32_t)(m >> 32), hi2 = hi << 1;
    asm("mad.lo.cc.u32 %0, %4, %4, %0;\n\t"
        "madc.hi.cc.u32 %1, %4, %4, %1;\n\t"
        "madc.lo.cc.u32 %2, %5, %5, %2;\n\t"
        "madc.hi.u32 %3, %5, %5, %3;\n\t"
        "mad.lo.cc.u32 %1, %4, %6, %1;\n\t"
        "madc.hi.cc.u32 %2, %4, %6, %2;\n\t"
        "addc.u32 %3, %3, 0;"
        : "+r"(a), "+r"(b), "+r"(c), "+r"(d)
        : "r"(lo), "r"(hi), "r"(hi2));
  }
  __device__ __forceinline__ u128 value() const {
    return ((u128)(((unsigned long long)d << 32) | c) << 64) | (((unsigned long long)b << 32) | a);
  }
};

// Squares of one loop's sums: W^2 to w2, C^2 + S^2 to f2, (T) Zr^2 + Zi^2 to z2.
template <bool T>
__device__ __forceinline__ void loop_squares(const long long *v, Sum128 &w2, Sum128 &f2, Sum128 &z2) {
  w2.add_square(v[0]);
  f2.add_square(v[1]);
  f2.add_square(v[2]);
  if (T) {
    z2.add_square(v[3]);
    z2.add_square(v[4]);
  }
}

// mul_q32 for v >= 0 and |c| <= 2^32 (its two 32-bit words, low first): with
// c = 2^32 M + l, floor((v c + 2^31) / 2^32) = M v + vh l + floor((vl l + 2^31) / 2^32).
__device__ __forceinline__ long long mul_len(long long v, int l, int M) {
  const uint32_t vl = (uint32_t)v, vh = (uint32_t)((unsigned long long)v >> 32), ul = (uint32_t)l;
  const unsigned long long t = (unsigned long long)vl * ul + 0x80000000ull;
  return (long long)((t >> 32) + (unsigned long long)vh * ul + (unsigned long long)((long long)M * v));
}

// Vertices of a tile whose ticks (and phase factors) the loop-properties
// kernel stages in shared memory; ticks beyond it are computed where needed.
constexpr int EST_STAGE = 1536;

// T: also the temporal moment (phase factors, Zr and Zi); off by default.
//
// Bound by instruction issue (74 % of the slots, 21 of 32 lanes active: the
// loop table's adds and the squares each take the lanes of their kind).  Flips
// come one bit per node (no root is followed for a flip), new operators leave
// as one bitmap word per warp and step, ticks take one conversion, lengths and
// squares 32-bit multiply-adds, the block's 128-bit sums warp reductions of 16-bit
// pieces: 0.86 -> 0.70 ms at L=16384, beta=4096 (790 -> 640 M warp instructions); of the instructions the table takes 22 %, the
// staging 15 %, the squares 10 %, the Fourier products 7 %.
template <int Q, bool T, int NT>
__global__ void __launch_bounds__(NT, (T ? 1536 : 2048) / NT) k_est(const DevChain *__restrict__ ch,
                                             const int2 *__restrict__ tab, int64_t blk0,
                                             Scratch s) {
  __shared__ int lkeys[LOOP_SLOTS];
  constexpr int NS = T ? LOOP_SUMS : 3;  // sums carried per loop
  __shared__ unsigned lvals[2 * NS * LOOP_SLOTS];
  __shared__ int4 csl[TILE], csr[TILE];  // 2^32 cos, 2^32 sin (low, high words) of a cell's two sites
  __shared__ char2 cx[TILE];             // cuts crossed by a leg that wraps, left and right
  extern __shared__ long long est_dyn[];
  long long *qv = est_dyn;                   // ticks q(tau) of the tile's vertices
  int2 *ev = (int2 *)(est_dyn + EST_STAGE);  // their phase factors exp(i w1 tau)
  __shared__ int stop;
  if (threadIdx.x == 0) stop = halted(s);
  const int64_t gt = blk0 + blockIdx.x;
  const int2 t = tab[gt];
  const DevChain &C = ch[t.x];
  const int c0 = t.y * TILE, c1 = min(C.ncell, c0 + TILE), ncl = c1 - c0;
  const int32_t *vp = s.vptr + C.cell_off;
  const int a = uniform(vp[c0]), e = uniform(vp[c1]);
  const int64_t vb = C.vtx_base, wb = vb >> 5;
  const int32_t *par = s.parent + vb;
  const uint64_t *vt = (const uint64_t *)s.vtau + vb;
  // A barrier of its own: with the answer taken at the one below (and the staging kept
  // in bounds whatever a and e are) 732 instead of 722 us at L=16384, beta=4096.
  __syncthreads();
  if (stop) return;
  const int F = C.F;
  // Ticks of every vertex of the tile, once: the fragments below a vertex
  // mostly start at vertices of the same tile.
  // Their phase factors too (temporal moment, w1 = 2 pi / beta).  They are
  // staged beside the cells' set-up, before the one barrier (behind a barrier
  // of their own the kernel took 0.866 ms instead of 0.854 at L=16384,
  // beta=4096).
  const uint64_t phR = C.phR;
  const int phS = C.phS;
  const int nq = min(min(e - a, local_cap(C)), EST_STAGE);
  const unsigned slot_mask =
      (C.loop_slots > 0 && C.loop_slots <= LOOP_SLOTS && !(C.loop_slots & (C.loop_slots - 1)))
          ? (unsigned)C.loop_slots - 1u
          : (unsigned)LOOP_SLOTS - 1u;
  for (int i = threadIdx.x; i < nq; i += blockDim.x) {
    const long long q = q_time(vt[a + i], F);
    qv[i] = q;
    if (T) ev[i] = phase_of((uint64_t)q, phR, phS, g_phase_tab);
  }
  if (threadIdx.x < ncl) {
    // per cell: Fourier weights of its two sites, cut crossings
    int b, j;
    cell_bj(C, c0 + threadIdx.x, b, j);
    const int ul = left_sub<Q>(b), ur = right_sub<Q>(b, C.L);
    const int xl = ul / Q, xr = ur / Q;
    const long long cl = C.cosq[xl], sl = C.sinq[xl], cr = C.cosq[xr], sr = C.sinq[xr];
    csl[threadIdx.x] = make_int4((int)cl, (int)(cl >> 32), (int)sl, (int)(sl >> 32));
    csr[threadIdx.x] = make_int4((int)cr, (int)(cr >> 32), (int)sr, (int)(sr >> 32));
    cx[threadIdx.x] = make_char2(s.cut_cross[C.sub_off + ul], s.cut_cross[C.sub_off + ur]);
  }
  for (int i = threadIdx.x; i < LOOP_SLOTS; i += blockDim.x) {
    lkeys[i] = -1;
#pragma unroll
    for (int k = 0; k < 2 * NS; ++k) lvals[2 * NS * i + k] = 0u;
  }
  __syncthreads();
  auto ticks = [&](int v) { return (unsigned)(v - a) < (unsigned)nq ? qv[v - a] : q_time(vt[v], F); };
  auto phase = [&](int v) {
    return (unsigned)(v - a) < (unsigned)nq ? ev[v - a]
                                            : phase_of((uint64_t)q_time(vt[v], F), phR, phS, g_phase_tab);
  };
  const uint32_t *flips = s.flipbits + wb;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // A warp takes a word of 32 vertices at a time and reconverges after it.
  // The flips and parents were written by an earlier kernel: they are read
  // through L1.
  Sum128 w2, f2, z2;  // this thread's share of the loops' squared sums
  long long newcnt = 0;
  for (int v0 = (a & ~31) + 32 * wid; v0 < e; v0 += NT) {
    const int w = v0 + lane;
    int nf = 0;
    if (w >= a && w < e) {
      const int ci = s.vcell[vb + w];
      const int P = s.pl[vb + w], R = s.pr[vb + w];
      const uint8_t f = s.vflag[vb + w];
      // an operator changes if the loops below and above it do not flip alike
      nf = (f ^ (flips[P >> 5] >> (P & 31)) ^ (flips[v0 >> 5] >> lane)) & VF_OLD;
      // fragment lengths in ticks of 2^-F: q(tau_top) - q(tau_bottom) (+ crossings)
      const long long qw = ticks(w);
      const long long qP = ticks(P);
      long long dl = qw - qP;
      long long dr = qw - (R == P ? qP : ticks(R));
      if (f & (VF_WRAP_L | VF_WRAP_R)) {
        const char2 x = cx[ci];
        if (f & VF_WRAP_L) dl += (long long)x.x * C.qbeta;
        if (f & VF_WRAP_R) dr += (long long)x.y * C.qbeta;
      }
      LoopSums x;
      x.v[0] = dl + dr;
      const int4 kl = csl[ci], kr = csr[ci];
      x.v[1] = mul_len(dl, kl.x, kl.y) + mul_len(dr, kr.x, kr.y);
      x.v[2] = mul_len(dl, kl.z, kl.w) + mul_len(dr, kr.z, kr.w);
      // int over a fragment of e^{i w1 t} dt = (e(top) - e(bottom)) / (i w1),
      // across the cut too (e(t + beta) = e(t)): both fragments end at w
      x.v[3] = x.v[4] = 0;
      if (T) {
        const int2 ew = phase(w), eP = phase(P), eR = (R == P) ? eP : phase(R);
        x.v[3] = 2ll * ew.x - eP.x - eR.x;
        x.v[4] = 2ll * ew.y - eP.y - eR.y;
      }
      if (P == R) {
        // Both upper legs of node P end at w, so P is a loop by itself and its
        // two fragments are the two below w: the loop's sums are complete here.
        loop_squares<T>(x.v, w2, f2, z2);
      } else {
        loop_add<NS>(lkeys, lvals, par[P], x, s, vb, slot_mask);
      }
    }
    const unsigned nm = __ballot_sync(0xffffffffu, nf);
    if (lane == 0) {
      newcnt += __popc(nm);
      store_word(s.newbits, wb + (v0 >> 5), nm, v0, a, e);
    }
  }
  __syncthreads();
  // A loop closed in the tile is complete in its slot: square it here.  A loop
  // that leaves the tile adds its slot to the root's global record, squared
  // once every tile has added (next operator list kernel).
  for (int h = threadIdx.x; h < LOOP_SLOTS; h += blockDim.x) {
    const int kk = lkeys[h];
    if (kk < 0) continue;
    long long v[LOOP_SUMS] = {};
#pragma unroll
    for (int i = 0; i < NS; ++i) v[i] = (long long)sget64(lvals + 2 * (NS * h + i));
    if (get_bit(s.openroot, wb, kk)) {
      acc_add<NS>(s, vb + kk, v);
    } else {
      loop_squares<T>(v, w2, f2, z2);
    }
  }
  u128 tw = w2.value(), tf = f2.value(), tz = T ? z2.value() : (u128)0;
  block_sums<T>(newcnt, tw, tf, tz);
  if (threadIdx.x == 0) {
    s.tile_sum2[gt] = newcnt;
    s.tile_sw2[2 * gt] = (unsigned long long)tw;
    s.tile_sw2[2 * gt + 1] = (unsigned long long)(tw >> 64);
    s.tile_sf2[2 * gt] = (unsigned long long)tf;
    s.tile_sf2[2 * gt + 1] = (unsigned long long)(tf >> 64);
    s.tile_sz2[2 * gt] = (unsigned long long)tz;
    s.tile_sz2[2 * gt + 1] = (unsigned long long)(tz >> 64);
  }
}

// ---- spins at tau = 0, vertex-free loops -------------------------------------------
// Site block gb: one thread per site (the threads past SITE_BLOCK have none).
// QT: Q = 2S if known at compile time, else 0.
template <int QT>
__device__ __forceinline__ void rewrite_sites(const DevChain *__restrict__ ch, const int2 *__restrict__ tab,
                                              int64_t gb, const Scratch &s) {
  const int2 t = tab[gb];
  const DevChain &C = ch[t.x];
  const int i = t.y * SITE_BLOCK + threadIdx.x, Q = QT ? QT : C.Q;
  const int64_t wb = C.vtx_base >> 5;
  long long nfree = 0;
  u128 w2 = 0, f2 = 0, none = 0;
  if (threadIdx.x < SITE_BLOCK && i < C.L) {
    const uint8_t *s0 = C.s0[C.cur];
    uint8_t *s1 = C.s0[C.cur ^ 1];
    for (int a = 0; a < Q; ++a) {
      const int u = i * Q + a;
      const int node = s.cut_node[C.sub_off + u];
      int f;
      if (node >= 0) {
        f = get_bit(s.flipbits, wb, node);
      } else {
        const int mn = s.free_min[C.sub_off + u];
        f = coin(C, TAG_FREE, (uint32_t)mn);
        if (mn == u) {
          ++nfree;
          const long long len = (long long)s.free_len[C.sub_off + u] * C.qbeta;
          w2 += sq_abs(len);
          f2 += sq_abs(mul_q32(len, C.cosq[i])) + sq_abs(mul_q32(len, C.sinq[i]));
        }
      }
      s1[u] = (uint8_t)(s0[u] ^ f);
    }
  }
  block_sums<false>(nfree, w2, f2, none);
  if (threadIdx.x == 0) {
    s.site_free[gb] = nfree;
    s.site_sw2[2 * gb] = (unsigned long long)w2;
    s.site_sw2[2 * gb + 1] = (unsigned long long)(w2 >> 64);
    s.site_sf2[2 * gb] = (unsigned long long)f2;
    s.site_sf2[2 * gb + 1] = (unsigned long long)(f2 >> 64);
  }
}

template <int Q>
__global__ void __launch_bounds__(SITE_BLOCK) k_sites(const DevChain *__restrict__ ch,
                                                      const int2 *__restrict__ tab, int64_t blk0,
                                                      Scratch s) {
  if (halted(s)) return;
  rewrite_sites<Q>(ch, tab, blk0 + blockIdx.x, s);
}

// ---- next operator list + open loops -------------------------------------------------
// The tile's new operators are a bitmap of its vertices: a scan of the words'
// counts gives every word's first place, a warp then moves the marked times of
// a word at a time (id order = order of the next operator list), and a cell's
// first operator is the count before its first vertex.
//
// Bound by the chain of dependent loads of a tile (table, chain, first vertices,
// words, then times and open roots), with 8 blocks per SM to hide it; more
// registers and fewer blocks lose (6 blocks 324 us).  So a tile passes two
// barriers only: a warp scans consecutive words of its own, which it then moves
// without a barrier, and the barrier of the final sums also covers the counts
// that the cells' offsets read.  The tile's own sums come in by cp.async
// meanwhile, and a warp takes the open roots of its words 32 at a time instead of
// a word's roots one after another.  L=16384, beta=4096 (32768 tiles): 277 -> 235
// us (249 with the sums read at the end); with the temporal sums, L=4098, beta=1000.7: 31 -> 25.
//
// SMALL (every chain has at most OWN_SCAN tiles): two launches less.  A tile
// adds up the counts before it itself instead of reading them from k_scan_ops,
// and the blocks past the ntiles tiles rewrite the site blocks' spins (k_sites),
// which need nothing of the operator list (with k_start's two parts in one launch:
// an update of the L=64 chain 55 -> 51 us, of L=1024, beta=256 93 -> 86 us;
// later steps brought these to 43 and 75).  Longer chains have the two kernels of their own: the code for both
// in one kernel cost the operator rewrite 4 % at 2^19 tiles (registers).  The line is
// set by the chain, not by the launch, and large batches of such chains lose by it:
// with half the blocks per SM the whole update takes 4 to 7 % more (ms, SMALL / the
// long chains' kernels: 16 chains of 25 tiles 0.116 / 0.121, 64 of 25 0.219 / 0.221,
// 4096 of one 0.730 / 0.750; 64 of 100 0.648 / 0.622, 512 of 100 4.56 / 4.29, 4096 of
// 100 35.8 / 33.6).
constexpr int OWN_SCAN = 1024;

template <bool T, bool SMALL>
__global__ void __launch_bounds__(TPB, T || SMALL ? 4 : 8) k_compact(DevChain *__restrict__ ch,
                                                 const int2 *__restrict__ tab, int64_t ntiles,
                                                 const int2 *__restrict__ site_tab, Scratch s) {
  constexpr int NW = TPB / 32;
  __shared__ uint32_t nbits[TPB];  // per word: new operators, and their number before it
  __shared__ int npre[TPB], wtot[NW];
  __shared__ uint32_t wsum[2][NW];
  __shared__ unsigned short olist[NW][32];
  __shared__ ulonglong2 tsum[3];
  const int2 t = SMALL && blockIdx.x >= ntiles ? make_int2(0, 0) : tab[blockIdx.x];
  // SMALL goes on past the one bit that it sets itself, a chain without room for its
  // operators: every thread then reads the same answer, and every chain's count is
  // taken.  (The updates enqueued behind such a one, whose other kernels return, come
  // here too.  They find its cell offsets and counts and empty bitmaps, and write to
  // the list that is not current, which the rerun writes again.)
  if ((__ldcg(s.status) & ~(SMALL ? ST_OP_OVERFLOW : 0)) != 0) return;
  if (SMALL && blockIdx.x >= ntiles) {
    rewrite_sites<0>(ch, site_tab, blockIdx.x - ntiles, s);
    return;
  }
  const int64_t gt = blockIdx.x;
  DevChain &C = ch[t.x];
  const int c0 = t.y * TILE, c1 = min(C.ncell, c0 + TILE), ncl = c1 - c0;
  const int32_t *vp = s.vptr + C.cell_off;
  const int64_t vb = C.vtx_base;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int64_t base = SMALL ? 0 : s.tile_pref2[gt];
  bool fits = true;
  if (SMALL) {
    uint32_t before = 0, all = 0;  // a chain has fewer than 2^31 operators
    for (int i = threadIdx.x; i < C.ntile; i += TPB) {
      const uint32_t x = (uint32_t)s.tile_sum2[C.tile0 + i];
      before += i < t.y ? x : 0u;
      all += x;
    }
    before = __reduce_add_sync(0xffffffffu, before);
    all = __reduce_add_sync(0xffffffffu, all);
    if (lane == 0) {
      wsum[0][wid] = before;
      wsum[1][wid] = all;
    }
  }
  const int a = uniform(vp[c0]), e = uniform(vp[c1]);
  const int cv = (threadIdx.x < ncl) ? vp[c0 + threadIdx.x] : e;  // first vertex of the thread's cell
  const int64_t wfirst = (vb + a) >> 5;
  const int nw = e > a ? (int)(((vb + e - 1) >> 5) - wfirst) + 1 : 0;
  // Words in chunks (one but for tiles of more than 8000 vertices); a warp takes
  // pw consecutive words of a chunk, one per lane.
  const int pw = max(1, min(32, (nw + NW - 1) / NW)), chunk = NW * pw;
  double *ntau = C.op_tau[C.cur ^ 1];
  if (threadIdx.x < (T ? 3 : 2)) {  // the sums that the tile's own loops left
    const unsigned long long *p = (threadIdx.x == 0 ? s.tile_sw2 : threadIdx.x == 1 ? s.tile_sf2 : s.tile_sz2) + 2 * gt;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(&tsum[threadIdx.x])), "l"(p) : "memory");
  }
  Sum128 sw, sf, sz;
  int run = 0, at = -1;  // new operators before the chunk; before the thread's cell
  auto cell_start = [&](int k0) {  // new operators before the cell's first vertex, if it lies in the chunk
    const int64_t k = ((vb + cv) >> 5) - wfirst - k0;
    if (cv < e && k >= 0 && k < chunk) at = npre[k] + __popc(nbits[k] & ((1u << (cv & 31)) - 1u));
  };
  for (int k0 = 0; k0 < nw || (SMALL && k0 == 0); k0 += chunk) {
    const int k = k0 + wid * pw + lane;
    const bool in = lane < pw && k < nw;
    uint32_t bits = 0u, open = 0u;
    if (in) {
      const int64_t wd = wfirst + k, v0 = (wd << 5) - vb;
      uint32_t mask = ~0u;
      if (v0 < a) mask &= ~0u << (a - v0);
      if (v0 + 32 > e) mask &= (e - v0 >= 32) ? ~0u : ((1u << (e - v0)) - 1u);
      bits = s.newbits[wd] & mask;
      open = __ldcg(s.openroot + wd) & mask;
    }
    const int cnt = __popc(bits);
    int inc = cnt, oinc = __popc(open);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, inc, o), z = __shfl_up_sync(0xffffffffu, oinc, o);
      if (lane >= o) {
        inc += y;
        oinc += z;
      }
    }
    if (lane == 31) wtot[wid] = inc;
    __syncthreads();
    if (SMALL && k0 == 0) {
      base = __reduce_add_sync(0xffffffffu, lane < NW ? wsum[0][lane] : 0u);
      const int64_t all = __reduce_add_sync(0xffffffffu, lane < NW ? wsum[1][lane] : 0u);
      fits = all <= C.op_cap;  // else no list is written: the host grows it and replays
      if (threadIdx.x == 0 && t.y == C.ntile - 1) {
        C.n_off_new = all;
        if (!fits) atomicOr(s.status, ST_OP_OVERFLOW);
      }
    }
    const int wt = lane < NW ? wtot[lane] : 0;
    const int pre = run + __reduce_add_sync(0xffffffffu, lane < wid ? wt : 0) + inc - cnt;
    run += __reduce_add_sync(0xffffffffu, wt);
    if (in) {
      nbits[k - k0] = bits;
      npre[k - k0] = pre;
    }
    const int64_t v0 = (wfirst + k0 + wid * pw) << 5;
    for (int i = 0; i < pw; ++i) {
      const uint32_t x = __shfl_sync(0xffffffffu, bits, i);
      const int p = __shfl_sync(0xffffffffu, pre, i);
      if (((x >> lane) & 1u) && fits) ntau[base + p + __popc(x & ((1u << lane) - 1u))] = s.vtau[v0 + 32 * i + lane];
    }
    // Loops that left their tile: one 32-byte record per root (and its Zi word),
    // read and cleared.  The roots cluster at a tile's first vertices: the warp
    // lists those of its words and takes one per lane.
    const int nopen = __shfl_sync(0xffffffffu, oinc, 31);
    for (int r0 = 0; r0 < nopen; r0 += 32) {
      int p = oinc - __popc(open) - r0;
      for (uint32_t x = open; x; x &= x - 1, ++p)
        if (p >= 0 && p < 32) olist[wid][p] = (unsigned short)(32 * lane + __ffs(x) - 1);
      __syncwarp();
      if (lane < nopen - r0) {
        const int64_t v = v0 + olist[wid][lane];
        const ulonglong2 x = s.acc2[2 * v], y = s.acc2[2 * v + 1];
        const unsigned long long zi = T ? s.accz[v] : 0ull;
        // The stores follow the loads' arrival (the sums are far below 2^63, so
        // the test always holds): issued with the loads still on their way to
        // the same sector, they made this kernel four times slower.
        if (((long long)x.x >= 0) & (y.x != 1ull << 63) & (zi != 1ull << 63)) {
          s.acc2[2 * v] = make_ulonglong2(0ull, 0ull);
          s.acc2[2 * v + 1] = make_ulonglong2(0ull, 0ull);
          if (T) s.accz[v] = 0ull;
        }
        sw.add_square((long long)x.x);
        sf.add_square((long long)x.y);
        sf.add_square((long long)y.x);
        if (T) {
          sz.add_square((long long)y.y);
          sz.add_square((long long)zi);
        }
      }
      __syncwarp();
    }
    if (nw > chunk) {  // the words' counts are overwritten by the next chunk
      __syncthreads();
      cell_start(k0);
      __syncthreads();
    }
  }
  long long none = 0;
  u128 w2 = sw.value(), f2 = sf.value(), z2 = T ? sz.value() : (u128)0;
  asm volatile("cp.async.wait_all;" ::: "memory");
  block_sums<T, true>(none, w2, f2, z2);  // its barrier also completes the words' counts
  if (nw && nw <= chunk) cell_start(0);
  int32_t *nptr = C.op_ptr[C.cur ^ 1];
  if (threadIdx.x < ncl) {
    nptr[c0 + threadIdx.x] = (int32_t)(base + (at < 0 ? run : at));
    // the last tile's operators end the list
    if (c0 + (int)threadIdx.x == C.ncell - 1) nptr[C.ncell] = (int32_t)(base + run);
  }
  if (threadIdx.x == 0) {
    auto add = [&](unsigned long long *t, const ulonglong2 &old, u128 v) {
      const u128 x = (((u128)old.y << 64) | old.x) + v;
      *(ulonglong2 *)(t + 2 * gt) = make_ulonglong2((unsigned long long)x, (unsigned long long)(x >> 64));
    };
    add(s.tile_sw2, tsum[0], w2);
    add(s.tile_sf2, tsum[1], f2);
    if (T) add(s.tile_sz2, tsum[2], z2);
  }
}

// ---- per-chain record -----------------------------------------------------------------
// A chain's tiles and site blocks in gridDim.y parts; each part leaves its sums
// at its first tile, and the part that finishes last adds them up and writes
// the record.  A chain of few tiles is one part, and its time is the chain of
// fp64 operations behind the sums (they are slow on GB300): the record's values
// and running sums are taken side by side, one per lane, with the loads they need
// issued beside the sums (launch 13 -> 8 us; one thread took them one after
// another).  One part per chain took 0.34 ms at 2^19 tiles.
struct ChainSums {
  long long roots, nfree;
  u128 w2, f2, z2;
};

__device__ __forceinline__ void add_sums(ChainSums &x, const ChainSums &y) {
  x.roots += y.roots;
  x.nfree += y.nfree;
  x.w2 += y.w2;
  x.f2 += y.f2;
  x.z2 += y.z2;
}

__device__ __forceinline__ u128 pair128(const unsigned long long *t, int64_t g) {
  return ((u128)__ldcg(t + 2 * g + 1) << 64) | __ldcg(t + 2 * g);
}

__device__ __forceinline__ void warp_sums(ChainSums &x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ChainSums y;
    y.roots = __shfl_down_sync(0xffffffffu, x.roots, o);
    y.nfree = __shfl_down_sync(0xffffffffu, x.nfree, o);
    y.w2 = shfl_down_u128(x.w2, o);
    y.f2 = shfl_down_u128(x.f2, o);
    y.z2 = shfl_down_u128(x.z2, o);
    add_sums(x, y);
  }
}

constexpr int FINAL_THREADS = 256;
constexpr int FINAL_BLOCKS = 152 * 16;  // of a launch, when chains are cut in parts

__global__ void __launch_bounds__(FINAL_THREADS) k_final(DevChain *__restrict__ ch, Scratch s) {
  __shared__ ChainSums part[FINAL_THREADS / 32];
  __shared__ int last;
  if (halted(s)) return;
  DevChain &C = ch[blockIdx.x];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, np = gridDim.y;
  const int per = (C.ntile + np - 1) / np, i0 = min(C.ntile, (int)blockIdx.y * per), i1 = min(C.ntile, i0 + per);
  const int pers = (C.nsiteblk + np - 1) / np, j0 = min(C.nsiteblk, (int)blockIdx.y * pers),
            j1 = min(C.nsiteblk, j0 + pers);
  // (nsiteblk <= ntile / k with k = ntile per site block, rounded up: a part
  // with site blocks has tiles)
  // What the record needs besides the sums, loaded beside them, for the block
  // that comes to write it.
  double run = 0.0, run2 = 0.0;
  if (threadIdx.x < NOBS) {
    run = C.sum[threadIdx.x];
    run2 = C.sumsq[threadIdx.x];
  }
  const int64_t n = C.n, n_new = C.n_off_new;
  const int32_t n_old = wid ? 0 : C.op_ptr[C.cur][C.ncell];
  lcqmc_record &r = C.ring[(uint64_t)C.n_rec % (uint32_t)C.ring_cap];
  ChainSums x{0, 0, 0, 0, 0};  // vertex-free loops are whole periods: no temporal term
  const int nt = i1 - i0, ns = j1 - j0;
  auto tile = [&](int64_t g) {
    return ChainSums{s.tile_roots[g], 0, pair128(s.tile_sw2, g), pair128(s.tile_sf2, g), pair128(s.tile_sz2, g)};
  };
  auto site = [&](int64_t g) {
    return ChainSums{0, s.site_free[g], pair128(s.site_sw2, g), pair128(s.site_sf2, g), 0};
  };
  if (nt + ns <= 32) {  // one warp takes them all
    if (wid) return;
    if (lane < nt)
      x = tile(C.tile0 + i0 + lane);
    else if (lane < nt + ns)
      x = site(C.site0 + j0 + lane - nt);
    warp_sums(x);
  } else {
#pragma unroll 4
    for (int i = i0 + threadIdx.x; i < i1; i += FINAL_THREADS) add_sums(x, tile(C.tile0 + i));
    for (int j = j0 + threadIdx.x; j < j1; j += FINAL_THREADS) add_sums(x, site(C.site0 + j));
    warp_sums(x);
    if (lane == 0) part[wid] = x;
    __syncthreads();
    if (wid) return;
    x = lane < FINAL_THREADS / 32 ? part[lane] : ChainSums{0, 0, 0, 0, 0};
    warp_sums(x);
  }
  if (np > 1) {  // this part's sums to its first tile's place (read by this block only)
    if (lane == 0) {
      if (i0 < i1) {
        const int64_t g = C.tile0 + i0;
        s.tile_roots[g] = x.roots;
        s.tile_sum2[g] = x.nfree;
        s.tile_sw2[2 * g] = (unsigned long long)x.w2;
        s.tile_sw2[2 * g + 1] = (unsigned long long)(x.w2 >> 64);
        s.tile_sf2[2 * g] = (unsigned long long)x.f2;
        s.tile_sf2[2 * g + 1] = (unsigned long long)(x.f2 >> 64);
        s.tile_sz2[2 * g] = (unsigned long long)x.z2;
        s.tile_sz2[2 * g + 1] = (unsigned long long)(x.z2 >> 64);
      }
      __threadfence();
      last = atomicAdd(s.part_done + blockIdx.x, 1u) == (unsigned)np - 1;
      __threadfence();
    }
    __syncwarp();
    if (!last) return;
    x = ChainSums{0, 0, 0, 0, 0};
    for (int p = lane; p < np; p += 32) {
      if (p * per >= C.ntile) break;
      const int64_t g = C.tile0 + (int64_t)p * per;
      add_sums(x, ChainSums{__ldcg((const long long *)s.tile_roots + g), __ldcg((const long long *)s.tile_sum2 + g),
                            pair128(s.tile_sw2, g), pair128(s.tile_sf2, g), pair128(s.tile_sz2, g)});
    }
    __syncwarp();
    warp_sums(x);
  }
  // lane 0 holds the chain's sums
  const int64_t n_free = __shfl_sync(0xffffffffu, x.nfree, 0),
                clusters = __shfl_sync(0xffffffffu, x.roots, 0) + n_free, n_seg = 2 * n + n_free;
  if (lane == 0) {
    r.n = n;
    r.n_off_old = n_old;
    r.n_off_new = n_new;
    r.n_free = n_free;
    r.n_clusters = clusters;
    r.n_seg = n_seg;
    r.F = C.F;
    r.pad = 0;
    r.sw2_lo = (unsigned long long)x.w2;
    r.sw2_hi = (unsigned long long)(x.w2 >> 64);
    r.sf2_lo = (unsigned long long)x.f2;
    r.sf2_hi = (unsigned long long)(x.f2 >> 64);
    r.sz2_lo = (unsigned long long)x.z2;
    r.sz2_hi = (unsigned long long)(x.z2 >> 64);
  }
  // Lanes 0, 1, 2, 8: energy, chi_s, chi_q, chi_w as numerator / denominator;
  // the other lanes below NOBS: whole numbers.
  //   energy = Q^2 J / 4 - n / (beta L);  chi = sum 2^-2F / (4 beta L)
  //   |int e^{i w1 t} dt|^2 = |Z|^2 2^-60 / w1^2 with w1 = 2 pi / beta:
  //   chi_w = sz2 2^-60 beta / (16 pi^2 L)
  unsigned long long lo, hi;
  {
    const unsigned long long wl = __shfl_sync(0xffffffffu, (unsigned long long)x.w2, 0),
                             wh = __shfl_sync(0xffffffffu, (unsigned long long)(x.w2 >> 64), 0),
                             fl = __shfl_sync(0xffffffffu, (unsigned long long)x.f2, 0),
                             fh = __shfl_sync(0xffffffffu, (unsigned long long)(x.f2 >> 64), 0),
                             zl = __shfl_sync(0xffffffffu, (unsigned long long)x.z2, 0),
                             zh = __shfl_sync(0xffffffffu, (unsigned long long)(x.z2 >> 64), 0);
    lo = lane == 1 ? wl : (lane == 2 ? fl : zl);
    hi = lane == 1 ? wh : (lane == 2 ? fh : zh);
  }
  double v = 0.0;
  if (lane < 3 || lane == 8) {
    const double two64 = 18446744073709551616.0, kPi = 3.14159265358979323846;
    const double L = (double)C.L;
    // 2^-2F and 2^-60: exact factors
    const double scale = __longlong_as_double((long long)(1023 - (lane == 8 ? 60 : 2 * C.F)) << 52);
    double num = (double)n, den = __dmul_rn(C.beta, L);
    if (lane) {
      num = __dmul_rn(__dadd_rn(__dmul_rn((double)hi, two64), (double)lo), scale);
      den = __dmul_rn(__dmul_rn(4.0, C.beta), L);
    }
    if (lane == 8) {
      num = __dmul_rn(num, C.beta);
      den = __dmul_rn(__dmul_rn(__dmul_rn(16.0, kPi), kPi), L);
    }
    v = __ddiv_rn(num, den);
    if (lane == 0) v = __dsub_rn(__dmul_rn(__dmul_rn((double)(C.Q * C.Q), C.J), 0.25), v);
  } else if (lane < NOBS) {
    const int64_t k = lane == 3 ? n : lane == 4 ? n_new : lane == 5 ? n_seg : lane == 6 ? clusters : n_seg + 2 * n;
    v = (double)k;
  }
  if (lane == 0) r.energy = v;
  if (lane == 1) r.chi_s = v;
  if (lane == 2) r.chi_q = v;
  if (lane == 8) r.chi_w = v;
  if (lane < NOBS) {
    C.sum[lane] = __dadd_rn(run, v);
    C.sumsq[lane] = __dadd_rn(run2, __dmul_rn(v, v));
  }
  __syncwarp();
  if (lane == 0) {
    if (np > 1) s.part_done[blockIdx.x] = 0;
    C.n_rec += 1;
    C.n_updates += 1;
    C.cur ^= 1;
    C.sweep += 1;
  }
}

// ---- host-side launchers ----------------------------------------------------------------
void set_full_table(const uint64_t *T, cudaStream_t st) {
  cudaMemcpyToSymbolAsync(c_T_full, T, sizeof(uint64_t) * KMAX, 0, cudaMemcpyHostToDevice, st);
}

static inline dim3 g1(int64_t n) { return dim3((unsigned)n); }

// One launch per Q group (Q = 2S = 1 .. QMAX); the tile-wide kernels that do
// not depend on Q run over the tiles of every group at once.
#define FOR_EACH_Q(M) M(1) M(2) M(3) M(4)
static_assert(QMAX == 4, "FOR_EACH_Q lists every Q");

static int64_t all_tiles(const Launch &L) {
  int64_t n = 0;
  for (int q = 0; q < QMAX; ++q) n += L.ntile[q];
  return n;
}

// Whether Q group q is launched: the one asked for, or all (only < 0).
static bool picked(int only, int q) { return only < 0 || only == q; }

int tunable(const Launch &L) {
  int used = all_tiles(L) <= WIDE_TILES ? 0 : TUNE_LINK | TUNE_COMPRESS;
  for (int q = 0; q < QMAX; ++q)
    if (L.ntile[q] > xt_max_tiles(q + 1)) used |= TUNE_LINK_X;
  return used;
}

void launch_start(const Launch &L, int64_t ntile, int64_t nw, cudaStream_t st) {
  int64_t nbb = 0;
  for (int q = 0; q < QMAX; ++q) nbb += L.nbondblk[q];
  const int64_t n = std::max<int64_t>(std::max(ntile, nw), SCAN_PARTS);
  const int64_t blocks = std::min<int64_t>((n + BOND_BLOCK - 1) / BOND_BLOCK, 152 * 16);
  k_start<<<g1(nbb + blocks), BOND_BLOCK, 0, st>>>(L.ch, L.bond_tab, nbb, L.s, ntile, nw);
}

void launch_insert(const Launch &L, int only, cudaStream_t st) {
  const bool wide = all_tiles(L) <= WIDE_TILES;
#define INSERT_QW(Q, NW)                                                                            \
  k_insert<Q, NW><<<g1(L.ntile[Q - 1]), 32 * NW, sizeof(InsSmem<Q, NW>), st>>>(L.ch, L.tile_tab,     \
                                                                              L.tile0[Q - 1], Q - 1, L.s)
#define INSERT_Q(Q)                              \
  if (L.ntile[Q - 1] && picked(only, Q - 1)) {   \
    if (wide)                                    \
      INSERT_QW(Q, INS_WARPS_WIDE);              \
    else                                         \
      INSERT_QW(Q, INS_WARPS);                   \
  }
  FOR_EACH_Q(INSERT_Q)
#undef INSERT_Q
#undef INSERT_QW
}

// Whether the operator rewrite adds up the tiles' counts by itself.
static bool own_scan(const Launch &L) { return L.max_ntile <= OWN_SCAN; }

void launch_scan_ops(const Launch &L, cudaStream_t st) {
  if (own_scan(L)) return;
  // Parts of at least 1024 tiles, and no more than one block per SM in all, so
  // that every part is resident while others wait for it.
  const int parts = (int)std::max<int64_t>(1, std::min<int64_t>(L.max_ntile / 1024, SCAN_PARTS / L.nchains));
  k_scan_ops<<<dim3(L.nchains, parts), 1024, 0, st>>>(L.ch, L.s);
}

void launch_cut(const Launch &L, int only, cudaStream_t st) {
#define CUT_Q(Q) \
  if (L.nsiteblk[Q - 1] && picked(only, Q - 1)) \
    k_cut<Q><<<g1(L.nsiteblk[Q - 1]), SITE_BLOCK * Q, 0, st>>>(L.ch, L.site_tab, L.site0[Q - 1], L.s);
  FOR_EACH_Q(CUT_Q)
#undef CUT_Q
}

void launch_link(const Launch &L, int only, cudaStream_t st) {
  const bool wide = all_tiles(L) <= WIDE_TILES;
#define LINK_Q(Q)                                                                                              \
  if (L.ntile[Q - 1] && picked(only, Q - 1)) {                                                                 \
    if (wide)                                                                                                  \
      k_link<Q, TPB_WIDE><<<g1(L.ntile[Q - 1]), TPB_WIDE, 0, st>>>(L.ch, L.tile_tab, L.tile0[Q - 1], L.s);      \
    else                                                                                                       \
      k_link<Q, TPB><<<g1(L.ntile[Q - 1]), L.link_threads, 0, st>>>(L.ch, L.tile_tab, L.tile0[Q - 1], L.s);     \
  }
  FOR_EACH_Q(LINK_Q)
#undef LINK_Q
  // Tile-crossing edges: a block per tile for few tiles, else a warp per tile.
  const int wpb = L.link_x_warps;
  for (int q = 0; q < QMAX; ++q) {
    const int64_t n = L.ntile[q];
    if (!n || !picked(only, q)) continue;
    if (n > xt_max_tiles(q + 1))
      k_link_x<<<g1((n + wpb - 1) / wpb), 32 * wpb, 0, st>>>(L.ch, L.tile_tab + L.tile0[q], n, L.s);
    else
      k_link_xt<<<g1(n), TPB_X, 0, st>>>(L.ch, L.tile_tab, L.tile0[q], L.s);
  }
}

void launch_compress(const Launch &L, int only, cudaStream_t st) {
  const int64_t n = only < 0 ? all_tiles(L) : L.ntile[only], t0 = only < 0 ? 0 : L.tile0[only];
  if (!n) return;
  if (all_tiles(L) <= WIDE_TILES)
    k_compress<TPB_WIDE><<<g1(n), TPB_WIDE, 0, st>>>(L.ch, L.tile_tab, t0, L.s);
  else
    k_compress<TILE><<<g1(n), L.compress_threads, 0, st>>>(L.ch, L.tile_tab, t0, L.s);
}

void launch_check_forest(const Launch &L, cudaStream_t st) {
  const int64_t n = all_tiles(L);
  if (n) k_check_forest<<<g1(n), TILE, 0, st>>>(L.ch, L.tile_tab, L.s);
}

// Per-vertex staging of the loop-properties kernel: ticks and phase factors.
constexpr size_t EST_DYN_SMEM = EST_STAGE * (sizeof(long long) + sizeof(int2));

// Device tables and kernel attributes, set once per process and device: the
// phase factor table (cos and sin of 2 pi k / 2^16 rounded to 30 fractional
// bits) and the loop-properties kernel's shared memory size.
int init_kernel_attributes() {
  static std::mutex mu;
  static bool done[256];
  static int2 tab[(1 << PHASE_BITS) + 1];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return -1;
  std::lock_guard<std::mutex> lk(mu);
  if (done[dev]) return 0;
  for (int k = 0; k <= (1 << PHASE_BITS); ++k) {
    const double ang = (2.0 * M_PI * (double)k) / (double)(1 << PHASE_BITS);
    tab[k] = make_int2((int)std::llrint(std::ldexp(std::cos(ang), 30)),
                       (int)std::llrint(std::ldexp(std::sin(ang), 30)));
  }
  // waited for: other streams read the table
  if (cudaMemcpyToSymbolAsync(g_phase_tab, tab, sizeof(tab), 0, cudaMemcpyHostToDevice, cudaStreamLegacy) !=
          cudaSuccess ||
      cudaStreamSynchronize(cudaStreamLegacy) != cudaSuccess)
    return -1;
#define EST_ATTR_Q(Q)                                                                      \
  if (cudaFuncSetAttribute(k_est<Q, true, TPB>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                           (int)EST_DYN_SMEM) != cudaSuccess ||                              \
      cudaFuncSetAttribute(k_est<Q, true, TPB_WIDE>,                                         \
                           cudaFuncAttributeMaxDynamicSharedMemorySize,                      \
                           (int)EST_DYN_SMEM) != cudaSuccess)                                \
    return -1;
  FOR_EACH_Q(EST_ATTR_Q)
#undef EST_ATTR_Q
#define INS_ATTR_Q(Q)                                                                                       \
  if (cudaFuncSetAttribute(k_insert<Q, INS_WARPS>, cudaFuncAttributeMaxDynamicSharedMemorySize,               \
                           (int)sizeof(InsSmem<Q, INS_WARPS>)) != cudaSuccess ||                              \
      cudaFuncSetAttribute(k_insert<Q, INS_WARPS_WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize,          \
                           (int)sizeof(InsSmem<Q, INS_WARPS_WIDE>)) != cudaSuccess)                           \
    return -1;
  FOR_EACH_Q(INS_ATTR_Q)
#undef INS_ATTR_Q
  done[dev] = true;
  return 0;
}

void launch_est(const Launch &L, int only, cudaStream_t st) {
  // without the temporal moment only the ticks are staged
  const size_t dyn = L.temporal ? EST_DYN_SMEM : EST_STAGE * sizeof(long long);
  const bool wide = all_tiles(L) <= WIDE_TILES;
#define EST_QTN(Q, T, NT) \
  k_est<Q, T, NT><<<g1(L.ntile[Q - 1]), NT, dyn, st>>>(L.ch, L.tile_tab, L.tile0[Q - 1], L.s)
#define EST_Q(Q)                               \
  if (L.ntile[Q - 1] && picked(only, Q - 1)) { \
    if (L.temporal && wide)                    \
      EST_QTN(Q, true, TPB_WIDE);              \
    else if (L.temporal)                       \
      EST_QTN(Q, true, TPB);                   \
    else if (wide)                             \
      EST_QTN(Q, false, TPB_WIDE);             \
    else                                       \
      EST_QTN(Q, false, TPB);                  \
  }
  FOR_EACH_Q(EST_Q)
#undef EST_Q
#undef EST_QTN
}

void launch_compact(const Launch &L, bool sites, cudaStream_t st) {
  const int64_t nt = all_tiles(L);
  if (own_scan(L)) {
    int64_t ns = 0;
    for (int q = 0; q < QMAX && sites; ++q) ns += L.nsiteblk[q];
    if (L.temporal)
      k_compact<true, true><<<g1(nt + ns), TPB, 0, st>>>(L.ch, L.tile_tab, nt, L.site_tab, L.s);
    else
      k_compact<false, true><<<g1(nt + ns), TPB, 0, st>>>(L.ch, L.tile_tab, nt, L.site_tab, L.s);
    return;
  }
  if (L.temporal)
    k_compact<true, false><<<g1(nt), TPB, 0, st>>>(L.ch, L.tile_tab, nt, L.site_tab, L.s);
  else
    k_compact<false, false><<<g1(nt), TPB, 0, st>>>(L.ch, L.tile_tab, nt, L.site_tab, L.s);
  if (sites) launch_sites(L, st);
}

void launch_sites(const Launch &L, cudaStream_t st) {
#define SITES_Q(Q) \
  if (L.nsiteblk[Q - 1]) k_sites<Q><<<g1(L.nsiteblk[Q - 1]), SITE_BLOCK, 0, st>>>(L.ch, L.site_tab, L.site0[Q - 1], L.s);
  FOR_EACH_Q(SITES_Q)
#undef SITES_Q
}

void launch_final(const Launch &L, cudaStream_t st) {
  // Parts of at least 512 tiles, and no more blocks in all than the chip holds a few
  // times over: every chain gets as many parts as the largest.  One chain of 32768
  // tiles with 16, 1024, 4096, 12000 chains of 8, 4, 1, 1 tiles, ms per update: 64
  // parts each 2.78, 3.34, 4.40, 7.47; so limited 2.78, 3.17, 3.50, 4.63.
  const int parts = (int)std::max<int64_t>(
      1, std::min<int64_t>(L.max_ntile / 512, std::min<int64_t>(64, FINAL_BLOCKS / L.nchains)));
  k_final<<<dim3(L.nchains, parts), FINAL_THREADS, 0, st>>>(L.ch, L.s);
}

}  // namespace lcq
