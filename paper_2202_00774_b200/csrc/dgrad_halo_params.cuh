// Launch parameters of the whole-filter-reuse data-gradient kernel.
#pragma once
#include "dgrad_common.cuh"

namespace sdgp {

constexpr int kHaloRows = 16;  // 8-pixel rows of a strip: the 128 rows of an accumulator

// Division by a divisor fixed for the launch: m = floor(2^32 / d) (0xFFFFFFFF for d = 1) gives a quotient
// that is at most one too small for any 32-bit x; one correction step makes it exact.
__host__ __device__ inline uint32_t div_magic(uint32_t d) { return d <= 1 ? 0xFFFFFFFFu : (uint32_t)(0x100000000ull / d); }
__device__ __forceinline__ void divmod(uint32_t x, uint32_t d, uint32_t m, uint32_t& q, uint32_t& r) {
  q = __umulhi(x, m);
  r = x - q * d;
  if (r >= d) { ++q; r -= d; }
}

// One output parity of a stride-2 convolution (or the whole of a stride-1 one): its filter taps, where they start, its pixels.
struct HaloClass {
  int R, S, sb;                          // sb: filter columns served by one box (see HaloParams)
  int pad_h, pad_w, r_first, s_first;
  int H, W;
};

struct HaloParams {
  int B, H, W, Cin, Cout;
  int R, S, pad_h, pad_w;
  int r_first, r_step, s_first, s_step, S_full;  // as in DgradParams
  int classes;             // 1, or 4: all output parities of a stride-2 convolution in one launch; R, S, H, W are then the largest
  int nt;                  // strips per CTA tile set (1 or 2), side by side, sharing every W stage
  int sets_w, tiles_h, tiles_n;
  int m_sets;              // sets_w * tiles_h * B
  uint32_t mg_tiles_n, mg_sets_w, mg_tiles_h;  // div_magic of the three counts above
  int pair_tiles;          // ceil(m_sets / 2) * tiles_n
  int units;               // work units: pair tiles, the last `units - split_from` of them split by strip
  int split_from;          // units >= split_from cover one strip of a pair tile each (quantisation of the last round)
  int k_blocks;
  int k_last, last_mmas;   // as in DgradParams
  int pitch;               // pixel columns of the A box: 8 * nt + S - 1
  int th, tb;              // a strip is 8 pixels wide and covers th pixel rows of tb images, th * tb = 16: 16 x 1, or 8 x 2
                           // for images at most 8 pixels tall. Its 16 rows are ordered (pixel row, image), so a vertical
                           // tap is still one uniform row offset (tb rows).
  int img_h;               // rows of the A box: (th + R - 1) * tb, ordered (pixel row, image)
  // Images 4 pixels wide: the 8 pixels of a strip row are the same pixel row of TWO images, a box row holds
  // img_per_row = 2 * nt images side by side with no column halo (an image's neighbour is another image), and
  // the horizontal taps are served by separate boxes: ss = S boxes per channel block, each fetched with its
  // own column offset (the tensor map zero-fills beyond an image's edge), sb = 1 filter column per box.
  // Otherwise img_per_row = 1, ss = 1, sb = S.
  int split, img_per_row, ss, sb;
  int k_uses;              // A boxes per tile set: k_blocks * ss
  int a_stages, a_shift;   // A ring depth (2 or 4) and its log2
  int img_rows;            // pitch * img_h
  // Fused mode, work units of the pruning warps (8 box pixels each). static_pad == 0: unit u = box pixels 8u .. 8u + 7
  // in row-major order, units_per_box = ceil(img_rows / 8). static_pad == 1 (a tile set spans its images from edge to
  // edge, so the halo rows and columns of EVERY box are padding): the stages are cleared once when the kernel starts and
  // only the units inside the images are ever pruned and written - unit u = 8 pixels from column unit_col0 + 8 * (u % nt)
  // of box row unit_row0 + u / nt, units_per_box = H * tb * nt. Fewer units per box also means fewer rounds of units
  // per pruning warp, which is what sets the time a box takes.
  int static_pad, units_per_box, unit_row0, unit_col0;
  int w_stages;
  int meta_col, meta_shared, out_bufs;
  int patch_store;         // not fused: strips are stored as TMA boxes by the four epilogue warps together (else rows)
  int a_bytes, eraw_bytes, w_bytes;  // per stage
  // Position metadata of an A box in the order the tensor core wants, stored ONCE per box and shared by every
  // tap: "master" pi (pi = 0, 1) pairs box rows (pi + 2m, pi + 2m + 1); its 16-byte line ((2m + e) * pitch + x)
  // holds, for the four MMAs of a channel block, the metadata of channels 16e .. 16e+15 of the MMA's 32 at
  // box pixel (pi + 2m, x) in the low half-words and of the pixel below it in the high half-words. The
  // TMEM image of tap (r, s) and strip j is then the window of 16 groups of 8 lines that starts at line
  // ((R-1-r - pi) * pitch + 8j + S-1-s) of master pi = (R-1-r) % 2, groups pitch lines apart: one
  // tcgen05.cp whose descriptor carries that start address and stride.
  int pairs0, pairs1;      // row pairs of the two masters
  int m0_bytes, meta_bytes;  // bytes of master 0; of both (one A stage)
  int off_eraw, off_meta, off_w, off_out, off_bar;
  int smem_bytes;
  // fused pruning (A is the dense dL/dO): the pruning warps read it straight from global memory
  const uint8_t* a_dense;  // dL/dO [B, P, Q, Cout], 16-bit elements
  int diag_cin_g, diag_cout_g, diag_last;  // grouped convolution: see first_k_block()
  uint32_t pitch_magic;    // ceil(2^20 / pitch): i / pitch == (i * pitch_magic) >> 20 for every box pixel row i
  int fused_n, fused_m, fused_scheme;
  uint32_t seed_lo, seed_hi;
  int P, Q;                // dO pixel grid (linear element index of the random scheme)
  OutView d;
  int last_launch, early;  // as in DgradParams
  int f16;                 // element type of A, W and dD: 0 = bf16, 1 = IEEE binary16
  // parity 2 * (row) + (column); classes == 1: cls[0] repeats the fields above (last: what every launch reads stays on fewer lines of parameters)
  HaloClass cls[4];
};

// dD's tensor maps: one, or one per parity.
template <bool CLASSES>
struct HaloOutMaps {
  CUtensorMap m[CLASSES ? 4 : 1];
};

// Plans and launches the kernel over BN = bn input channels and nt strips (two at most, 256 columns together) per tile;
// SDGP_ERR_UNSUPPORTED if no plan fits.
sdgp_status launch_halo_sparse(int bn, int nt, const void* A, const void* meta, const void* Wt, const DgradView& view, const HaloParams& p, cudaStream_t stream);
sdgp_status launch_halo_dense(int bn, int nt, const void* A, const void* Wt, const DgradView& view, const HaloParams& p, cudaStream_t stream);
sdgp_status launch_halo_fused(int bn, int nt, const void* dO, const void* Wt, const DgradView& view, const HaloParams& p, cudaStream_t stream);
// The same plans without a launch.
bool plan_halo_sparse(int bn, int nt, HaloParams* p);
bool plan_halo_dense(int bn, int nt, HaloParams* p);
cudaError_t take_error_halo_sparse(unsigned int* word);
cudaError_t take_error_halo_dense(unsigned int* word);
cudaError_t take_error_halo_fused(unsigned int* word);

}  // namespace sdgp
