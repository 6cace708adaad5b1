// Launch interface between the host engine and the update kernels.
#pragma once
#include "dev.cuh"

namespace lcq {

// One batch's launch geometry.  Tiles, site blocks and bond blocks are grouped
// by Q = 2S (every Q=1 chain's blocks first, then Q=2, ...); index [q]
// addresses the Q = q+1 group.
struct Launch {
  DevChain *ch;
  int nchains;
  int64_t max_ntile;  // tiles of the largest chain
  Scratch s;
  const int2 *tile_tab, *site_tab, *bond_tab;
  int64_t ntile[QMAX], tile0[QMAX];
  int64_t nsiteblk[QMAX], site0[QMAX];
  int64_t nbondblk[QMAX], bond0[QMAX];
  int temporal;  // measure the temporal moment chi(pi, 2 pi / beta) too
  // block sizes of the union-find phases for launches of many tiles (any choice
  // gives the same results; few tiles: TPB_WIDE threads, k_link_xt)
  int link_threads = 256;     // k_link: 128 or 256
  int link_x_warps = 8;       // k_link_x: 1 .. 8 warps (one tile each) per block
  int compress_threads = 128; // k_compress: 32, 64, 96 or 128
  int check_forest = 0;       // verify the loop forest after compression (debug)
};

// Which of the three block sizes the launches use: TUNE_LINK | TUNE_LINK_X |
// TUNE_COMPRESS
enum : int { TUNE_LINK = 1, TUNE_LINK_X = 2, TUNE_COMPRESS = 4 };
int tunable(const Launch &L);
void set_full_table(const uint64_t *T, cudaStream_t st);
int init_kernel_attributes();
// bond parities; zeroes the look-back words of ntile tiles, the tickets and nw
// words of each bitmap
void launch_start(const Launch &L, int64_t ntile, int64_t nw, cudaStream_t st);
// only: the Q group to launch (Q - 1), or -1 for all of them
void launch_insert(const Launch &L, int only, cudaStream_t st);
void launch_scan_ops(const Launch &L, cudaStream_t st);
void launch_cut(const Launch &L, int only, cudaStream_t st);
void launch_link(const Launch &L, int only, cudaStream_t st);
void launch_compress(const Launch &L, int only, cudaStream_t st);
void launch_check_forest(const Launch &L, cudaStream_t st);
void launch_est(const Launch &L, int only, cudaStream_t st);
// operator rewrite; sites: the spin rewrite too, in the same launch where that
// is faster (else launch_sites is the caller's)
void launch_compact(const Launch &L, bool sites, cudaStream_t st);
void launch_sites(const Launch &L, cudaStream_t st);
void launch_final(const Launch &L, cudaStream_t st);

}  // namespace lcq
