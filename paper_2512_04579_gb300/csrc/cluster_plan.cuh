// cluster_plan.cuh -- layout and protocol arithmetic of the cluster Cholesky
// (chol_cluster.cuh): which CTA of a cluster owns which block rows, how much
// shared memory that takes, and which word reports a failed diagonal block.
// Plain C++ without CUDA types, so that the host compiler can build it for the
// CPU tests.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define GNM_HD __host__ __device__ __forceinline__
#else
#define GNM_HD inline
#endif

namespace gnm {

constexpr int kClBlock = 16;       // rows and columns of a block (the panel width of chol.cuh)
constexpr int kClMaxBlocks = 256;  // block rows of 16 an instance may have (n <= 4096; shared memory sets less)
constexpr int kClMaxRows = 32;     // block rows a rank may own (half warps of a CTA)

// Row plan entry of block row I (host-made, cluster_plan): owning rank and the
// index of the row's first block in the rank's block storage.
GNM_HD int cl_entry(int rank, int slot) { return (rank << 24) | slot; }
GNM_HD int cl_rank(int e) { return e >> 24; }
GNM_HD int cl_slot(int e) { return e & 0xFFFFFF; }

// Doubles of a CTA's shared memory ahead of its block rows.
GNM_HD int64_t cl_fixed_doubles(int n) { return 512 + 1024 + 256 + 68 + (int64_t)((n + 15) / 16) * 256; }

// Word in which rank 0 reports a failed diagonal block d, and that every rank
// reads behind the cluster barrier that ends panel d - 1.  Rank 0 may already be
// working on block d + 1 while another warp still is to read block d's word (no
// barrier of panel d has completed by then), so consecutive blocks use two
// words; the word of block d + 2 is block d's again, and its store follows
// panel d's second barrier, which the reader has arrived at.
GNM_HD int cl_fail_word(int d) { return d & 1; }

// Host side: row plans of an n x n system over cs ranks.  A block update (16^3
// DFMA) takes about 2600 cycles of an SM's FP64 pipe, rank 0's chain per panel
// 18600 (its 16 pivot columns run one after another, about 900 cycles each),
// seven block updates; so rank 0 starts with that load and the rows go, longest
// first, to the least loaded rank.
constexpr int kClChainBlocks = 7;
inline int cluster_plan(int n, int cs, int* plan) {  // returns the most blocks a rank stores
  const int nblk = (n + kClBlock - 1) / kClBlock;
  long load[16] = {0};
  int slots[16] = {0};
  load[0] = (long)kClChainBlocks * nblk;
  for (int I = nblk - 1; I >= 0; --I) {
    int q = 0;
    for (int k = 1; k < cs; ++k)
      if (load[k] < load[q]) q = k;
    plan[I] = cl_entry(q, slots[q]);
    slots[q] += I + 1;
    load[q] += (long)I * (I + 1) / 2 + 1;
  }
  int most = 0, rows[16] = {0};
  for (int I = 0; I < nblk; ++I)
    if (++rows[plan[I] >> 24] > kClMaxRows) return 1 << 20;
  for (int k = 0; k < cs; ++k) most = slots[k] > most ? slots[k] : most;
  return most;
}
// Block updates of the longest path through the factorisation (plan of n, cs).
inline long cluster_path(int n, int cs, const int* plan) {
  const int nblk = (n + kClBlock - 1) / kClBlock;
  (void)cs;
  long path = 0;
  for (int p = 0; p + 1 < nblk; ++p) {
    long load[16] = {kClChainBlocks};
    long worst = kClChainBlocks;
    for (int I = p + 2; I < nblk; ++I) {
      long& l = load[plan[I] >> 24];
      l += I - p;
      worst = l > worst ? l : worst;
    }
    path += worst + 2;  // + the panel's own blocks and the two barriers
  }
  return path;
}

}  // namespace gnm
