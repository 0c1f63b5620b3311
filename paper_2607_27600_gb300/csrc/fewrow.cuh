// fewrow.cuh -- interface of the GEMM for launches of few rows (short
// caches, small chunks, decode batches): gemm.cuh's products with the weight
// rows on the tensor cores' M side.
#pragma once
#include "gemm.cuh"

namespace cc {

constexpr int kFewMaxSplit = 8;   // CTAs of a cluster: K splits, or half as many of pairs (the portable size)

// How a launch is cut: row groups of nb activation rows (the N of a product),
// column tiles of 128 columns, and the K range of each tile over `split` CTAs
// of a cluster.
struct FewPlan {
  int nb, split;
  bool pair;       // two column tiles to a pair of CTAs, which share the activation rows
  int clusters;    // clusters of the launch at most: those resident at once
  int n_tiles;     // column tiles (EPI_QKV: those of Q, K and V, each rounded up)
  double cycles;   // estimated SM cycles
};

constexpr int kFewTileCols = 128;   // output columns of a tile
// Clusters of 2^i CTAs that a device holds at once, one CTA per SM: those of four and
// eight leave SMs of a GPC over (152 SMs: 76 of two, 36 of four and 15 of eight by the
// occupancy query).  From the SM count alone, not the query: which SMs are missing
// differs between devices, and a row's K split, so its bits, would with it.
struct FewClusters {
  int n[4];
};
FewClusters few_clusters(int sms);
// The plan for seqs sequences of at most rows_per_seq rows each.  row_pairs > 0:
// one group of 2 * row_pairs rows (GemmParams::row_pairs).
FewPlan few_plan(int epi, int n_tiles, int K, bool a_split, int seqs, long long rows_per_seq,
                 int row_pairs, const FewClusters &fit);
// The plan's estimated SM cycles where each sequence turns out to have rows_per_seq rows.
double few_cycles(const FewPlan &plan, int epi, int K, bool a_split, int seqs, long long rows_per_seq,
                  const FewClusters &fit);
// a: A rows x K, box 64 x plan.nb (half of it with pair); b (b2, b3): weights N x K, box 64 x 128, and
// for rotated projections (EPI_QROPE's b, EPI_QKV's b and b2) the 5-D view
// [heads][head_dim / 32][2][16][K], box {64, 16, 2, head_dim / 32, 128 / head_dim}.
// one_group: the launch has one row group (known on the host), so the first
// weight tiles are fetched before the previous kernel has finished.
cudaError_t launch_few(int epi, const CUtensorMap &a, const CUtensorMap &b, const CUtensorMap &b2,
                       const CUtensorMap &b3, const GemmParams &p, const FewPlan &plan,
                       bool one_group, cudaStream_t stream);

}  // namespace cc
