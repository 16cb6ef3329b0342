// Launch parameters of the general data-gradient kernel.
#pragma once
#include "dgrad_common.cuh"

namespace sdgp {

struct DgradParams {
  int B, H, W;            // dD pixel grid (fully connected: B = H = 1, W = rows)
  int Cin, Cout;
  int R, S;               // filter taps of this launch (stride 2: the taps of one output-parity class)
  int pad_h, pad_w;       // dO pixel of output pixel (h,w) under tap (r,s): (h + pad_h - r, w + pad_w - s)
  int r_first, r_step, s_first, s_step, S_full;  // tap (r,s) of the launch is filter tap (r_first + r_step*r, s_first + s_step*s)
  int TW, TH, TB;         // pixel patch of one CTA tile, TW * TH * TB <= 128
  int tiles_w, tiles_h, tiles_b, tiles_n;
  int m_tiles;            // tiles_w * tiles_h * tiles_b
  int pair_tiles;         // ceil(m_tiles / 2) * tiles_n
  int k_blocks;           // channel blocks per tap: ceil(Cout / channels per stage)
  int k_last, last_mmas;  // the layer's last channel block and the MMAs it needs (1..4)
  int rr;                 // vertical taps served by one A stage: 1, or R (filter-row reuse)
  int img_rows;           // pixel rows of one A stage: TW * (TH + rr - 1) * TB
  int stages;             // shared-memory pipeline depth
  int nacc;               // TMEM accumulators (2 = epilogue overlaps the next tile)
  int meta_col;           // first TMEM column of the metadata slots
  int meta_shared;        // metadata slots live in the first columns of the accumulator NOT being written
  int last_launch;        // no further launch of the same call follows
  int early;              // the next kernel may be scheduled while this one runs (early_for())
  int w_resident;         // whole W half-slice kept in shared memory
  int out_bufs;           // staging slabs per epilogue warp (boxes only)
  int box_store;          // the epilogue's warps write boxes of 32 pixels by TMA (else rows, straight from registers)
  // fused pruning (the kernel reads dense dL/dO and prunes it while staging A)
  int fused_n, fused_m, fused_scheme;
  uint32_t seed_lo, seed_hi;
  int P, Q;               // dO pixel grid (for the linear element index of the random scheme)
  OutView d;
  int f16;                // element type of A, W and dD: 0 = bf16, 1 = IEEE binary16
  // grouped convolution (block-diagonal W): a tile of input channels sees only k_blocks channel blocks of dL/dO,
  // starting at first_k_block(); diag_cin_g == 0: every tile sees all of them
  int diag_cin_g, diag_cout_g, diag_last;
  int off_raw;            // dense dL/dO stages: 2 * a_bytes each (two boxes of 64 channels)
  // shared-memory carve (byte offsets from the 1024-aligned base) and per-stage sizes
  int a_bytes, b_bytes, eraw_bytes, ehw_bytes;
  int off_b, off_eraw, off_ehw, off_w, off_out, off_bar;
  int smem_bytes;
};

// Plans and launches the kernel over BN = bn input channels per tile; SDGP_ERR_UNSUPPORTED if no plan fits.
sdgp_status launch_general(bool sparse, bool fused, int bn, const void* A, const void* meta, const void* Wt, const DgradView& view,
                           const DgradParams& p, cudaStream_t stream);
cudaError_t take_error_general(unsigned int* word);

}  // namespace sdgp
