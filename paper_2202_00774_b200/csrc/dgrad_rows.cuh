// Launch parameters of the fused prune + contraction kernel over rows (fully connected layers, 1 x 1 convolutions).
#pragma once
#include "dgrad_common.cuh"

namespace sdgp {

struct RowsParams {
  int rows, K, N;
  int n, m;
  uint32_t seed_lo, seed_hi;
  int f16;
  int k_blocks;            // blocks of 128 channels
  int last_mmas;           // MMAs (32 channels each) of the last block
  int n_tiles, n_groups, group_tiles;  // column tiles of BN; groups of them, whose accumulators are in TMEM together
  int works;               // row tiles of 256 x n_groups: what the CTA pairs take in turn
  int acc_ring;            // accumulators in TMEM, used in turn by the column tiles (the epilogue overlaps later tiles)
  int meta_col;            // first TMEM column of the metadata slots (four columns per A stage)
  int raw_stages, a_stages, w_stages;
  int off_a, off_meta, off_w, off_out, off_bar, smem_bytes;
};

struct RowsPlan {
  bool ok;
  int bn;
  double cost;  // estimated clocks
  RowsParams p;
};
// stage_clk: clocks the pruning warps take for a block of 128 channels. (Kept per thread for the last shapes asked for.)
RowsPlan plan_rows(int64_t rows, int K, int N, int stage_clk);

// dD [rows, N] = prune(dO [rows, K]) . W, pruned inside the kernel (n <= 2). W has w_rows >= K rows of w_cols >= N columns.
sdgp_status launch_rows_fused(const RowsPlan& plan, const void* dO, const void* W, int w_rows, int w_cols, void* dD,
                              const FusedPrune& prune, int dtype, cudaStream_t stream);
cudaError_t take_error_rows(unsigned int* word);

}  // namespace sdgp
