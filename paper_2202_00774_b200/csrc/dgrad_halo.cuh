// The whole-filter-reuse data-gradient kernel.
//
// Convolutions with more than one filter tap.
// The shared-memory matrix descriptor swizzles by absolute address bits, so an A operand may
// start at ANY 128-byte row of a swizzled tile and its 8-row groups may lie any number of rows
// apart. A tile is therefore a strip of 16 rows of 8 pixels, and one TMA box holding the strip plus
// its (R-1, S-1) halo serves EVERY filter tap: tap (r, s) is the row offset
// (R-1-r) * tb * pitch + (S-1-s) in the A descriptor, group stride = pitch rows. dL/dO is
// read from L2 once per strip (plus halo) instead of once per horizontal tap, and with two
// neighbouring strips per CTA (two accumulators) each W stage feeds twice the MMAs.
// Strip geometries (th pixel rows x tb images, th * tb = 16): 16 rows of one image; 8 rows of two images
// (images at most 8 pixels tall; the box's rows are ordered (pixel row, image)); and, for images 4 pixels
// wide, 4 rows of eight images with two images side by side in a strip row and one box per filter column
// (column-split mode: no column halo, five-dimensional tensor maps).
//
// Rings: A boxes (2 or 4 stages; one stage = one tile set and one block of output channels, with the raw
// metadata box TMA delivers and the two metadata masters built from it), W taps (w_stages; one stage = the W
// rows of one tap and channel block, and a slot of TMEM columns for that tap's metadata).
// Metadata masters: the position metadata of a box is stored once, in the order the tensor core wants, and every
// tap copies a window of it into TMEM (see HaloParams). Two-pass: warps 2..5 build the masters of each box;
// fused: the pruning warps write them directly.

#pragma once
#include "dgrad_halo_params.cuh"
#include "dgrad_prune.cuh"

namespace sdgp {
namespace {

constexpr int kHaloAStages = 4;  // at most: A stages in use are p.a_stages = 2, or 4 when the boxes are small (a power of two)
// Warp roles of the fused whole-filter-reuse kernel (24 warps: registers are granted to warps in fours, and
// 24 x 80 registers is what fits): warp 0 streams W, warp 1 issues the MMAs, warps 4..7 are the epilogue (one per
// TMEM lane quarter) and the other eighteen prune. Warp w runs on scheduler w % 4, so four pruning warps (9, 13, 17,
// 21) share the scheduler of the MMA-issuing warp; measured, their integer-pipe time is worth more than the issue
// slots they take from it (14 -> 16 -> 18 pruning warps: 1062 -> 1107 -> 1111 TFLOP/s on the ResNet-9 chain).
constexpr int kPruneWarps = 18;
constexpr int kThreadsHaloFused = 24 * 32;
// Not fused: one warp more than the general kernel's ten. It fetches the A boxes: with both in one warp W's loads waited for A's stages and A's
// for a place between W's (the MMA warp stood 100 to 130 clocks a tap for W, and a launch began with A before W). Us, prune
// kernel included: 64 -> 128 channels at 32 x 32, batch 512, 82.0 -> 75.0; 512 -> 512 at 4 x 4 (four boxes ahead) 22.9 -> 18.0; 64 x 7 x 7, 512 -> 512
// 17.2 -> 15.4; 256 -> 512 at 8 x 8 39.6 -> 37.6; 72 x 56 x 56, 192 -> 64, bound by stores, 69.4 -> 70.6.
constexpr int kABoxWarp = 10;
constexpr int kThreadsHalo = 11 * 32;

// PATCH (not fused): strips leave as one TMA box each (store_patch), else as rows; plan_halo() has the rule. Such a launch may also hold
// the four output parities of a stride-2 convolution (p.classes == 4): a work unit is then a tile set of one parity. The four of a
// tile are neighbouring units, so that its dL/dO comes from memory once and the pixels of dD that lie side by side are stored at
// about the same time; which of them falls to which CTA pair turns from tile to tile, for they have one, two, two and four taps. Us, 128 -> 128
// channels at 56 x 56, batch 256, random pruning included: four launches 104, this 92. Two kernels, so that neither carries the
// other's code.
template <bool SPARSE, int BN, int NT, bool FUSED, bool PATCH>
__global__ void __launch_bounds__(FUSED ? kThreadsHaloFused : kThreadsHalo, 1)
dgrad_halo_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmE,
                  const __grid_constant__ CUtensorMap tmB, const __grid_constant__ HaloOutMaps<PATCH> tmD,
                  const __grid_constant__ HaloParams p) {
  using C = Cfg<SPARSE, BN>;
  constexpr int kEpilogueWarp0 = FUSED ? 4 : 6;  // first of the four epilogue warps
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sA = smem;
  uint8_t* sEraw = smem + p.off_eraw;    // two-pass: the row-major metadata box as TMA delivers it
  uint8_t* sMeta = smem + p.off_meta;    // the two metadata masters of each A stage
  uint8_t* sW = smem + p.off_w;
  uint8_t* sOut = smem + p.off_out;
  uint64_t* a_full = (uint64_t*)(smem + p.off_bar);
  uint64_t* a_empty = a_full + kHaloAStages;
  uint64_t* meta_full = a_empty + kHaloAStages;
  uint64_t* meta_ready = meta_full + kHaloAStages;  // two-pass: the masters of the A stage are built (both CTAs)
  uint64_t* w_ready = meta_ready + kHaloAStages;    // W bytes landed
  uint64_t* w_empty = w_ready + kMaxStages;
  uint64_t* acc_full = w_empty + kMaxStages;
  uint64_t* acc_empty = acc_full + 2;
  uint64_t* meta_free = acc_empty + 2;
  uint32_t* tmem_slot = (uint32_t*)(meta_free + 2);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = ptx::cluster_ctarank();
  unsigned int* err = &g_device_error;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kHaloAStages; ++s) {
      // fused: A and its metadata rows are complete when every pruning warp has arrived
      // (a_full: the warps of both CTAs; meta_full: this CTA's)
      // (one arrival per work unit of the box: 8 pixel rows)
      ptx::mbar_init(&a_full[s], FUSED ? 2 * p.units_per_box : 1);
      ptx::mbar_init(&a_empty[s], 1);
      ptx::mbar_init(&meta_full[s], 1);
      ptx::mbar_init(&meta_ready[s], 8);  // four metadata warps in each CTA
    }
    for (int s = 0; s < kMaxStages; ++s) {
      ptx::mbar_init(&w_ready[s], 1);  // the producer's arrival with the byte count
      ptx::mbar_init(&w_empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      ptx::mbar_init(&acc_full[a], 1);
      ptx::mbar_init(&acc_empty[a], 8);
      ptx::mbar_init(&meta_free[a], 8);
    }
    ptx::fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    ptx::prefetch_tensormap(&tmA);
    ptx::prefetch_tensormap(&tmB);
    if (PATCH) ptx::prefetch_tensormap(&tmD.m[0]);
    if (SPARSE) ptx::prefetch_tensormap(&tmE);
  }
  if (warp == 1) {
    ptx::tmem_alloc_pair(tmem_slot, kTmemCols);
    ptx::tmem_relinquish_pair();
  }
  ptx::tc_fence_before_sync();
  ptx::cluster_sync();
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base_any = *tmem_slot;
  const uint32_t tmem_base = tmem_base_any;
  // everything above touched no global memory; the previous kernel's results are needed from here on
  ptx::wait_for_previous_grid();
  // Only now may the next kernel of the stream be scheduled: every CTA of this grid owns its TMEM
  // and has passed its cluster barrier and its wait for the previous grid, so a younger grid can
  // never sit between this grid and a resource it still needs, and at most one grid is resident
  // behind a running one. The younger grid's own TMEM allocation then simply waits for this grid
  // to free its columns, which it does without anyone's help.
  if (p.early) ptx::launch_dependents();

  const int pair_stride = gridDim.x >> 1;
  const int first_pair = blockIdx.x >> 1;
  // pair tile (p.classes == 4: and output parity) of unit number lt of this CTA
  auto unit_of = [&p, first_pair, pair_stride](int lt, int& c) -> int {
    c = 0;
    const int u = first_pair + lt * pair_stride;
    const int pt = u < p.split_from ? u : p.split_from + ((u - p.split_from) >> 1);
    if (!PATCH || p.classes == 1) return pt;
    c = (pt + (pt >> 2)) & 3;
    return pt >> 2;
  };
  auto class_of = [&p](int c) -> HaloClass {
    if (PATCH) return p.cls[c];
    return HaloClass{p.R, p.S, p.sb, p.pad_h, p.pad_w, p.r_first, p.s_first, p.H, p.W};
  };
  const int my_tiles = first_pair < p.units ? (p.units - first_pair + pair_stride - 1) / pair_stride : 0;
  const int n_half = (int)rank * C::kBCols;
  constexpr int set_cols = NT * BN;  // TMEM columns of one tile set's accumulators
  const int WS = p.w_stages;
  // Work unit u: a pair tile, or - for the units of the last, partly filled round - one strip of
  // a pair tile, so that the round costs half. strip_mask: the strips unit number lt of this CTA covers.
  auto strip_mask = [&p, first_pair, pair_stride](int lt) -> uint32_t {
    const int u = first_pair + lt * pair_stride;
    return u < p.split_from ? ((1u << NT) - 1u) : (1u << ((u - p.split_from) & 1));
  };
  // tile set of unit number lt for this CTA: first input channel, first pixel column / row, image; its parity
  auto locate = [&p, rank, &unit_of](int lt, int& n0, int& w0, int& h0, int& b0, int& c) -> bool {
    const int pt = unit_of(lt, c);
    uint32_t q, r;
    divmod((uint32_t)pt, (uint32_t)p.tiles_n, p.mg_tiles_n, q, r);
    n0 = (int)r * BN;
    const uint32_t t = 2u * q + rank;
    const bool in_range = (int)t < p.m_sets;  // a set past the last one loads zeros and stores nothing
    divmod(t, (uint32_t)p.sets_w, p.mg_sets_w, q, r);
    w0 = (int)r * 8 * NT;
    divmod(q, (uint32_t)p.tiles_h, p.mg_tiles_h, q, r);
    h0 = (int)r * p.th;
    b0 = (int)q * p.tb * p.img_per_row;
    return in_range;
  };

  if (!FUSED && warp == kABoxWarp) {
    // ------------------------------------------------------------ A boxes and their raw metadata
    if (ptx::elect_one()) {
      const uint32_t a_tx = 2u * (uint32_t)(p.img_rows * 128);
      const uint32_t meta_tx = (uint32_t)(p.img_rows * 16);
      bool alive = true;
      int ast = 0;
      uint32_t aph = 0;
      for (int lt = 0; alive && lt < my_tiles; ++lt) {
        int n0, w0, h0, b0, c;
        locate(lt, n0, w0, h0, b0, c);
        const int kb0 = first_k_block(p, n0, C::kKB);
        const HaloClass cl = class_of(c);
        const int p0 = h0 + cl.pad_h - (cl.R - 1), bg = b0 / p.img_per_row;
        for (int ku = 0; ku < p.k_uses; ++ku) {
          const int kl = ku / p.ss, si = ku - kl * p.ss;  // channel block of the tile's window, filter column of the box (column-split mode)
          const int kb = kb0 + kl, q0 = w0 + cl.pad_w - (cl.sb - 1) - si;
          if (!ptx::mbar_wait<kIdleWaitNs>(&a_empty[ast], aph ^ 1u, err, 0x100u + ast)) { alive = false; break; }
          // coordinates: channel, pixel column, image within a box row, image group, pixel row
          // (the tensor maps have the image-within-row dimension only in column-split mode)
          if (rank == 0) ptx::mbar_arrive_expect_tx(&a_full[ast], a_tx);
          if (SPARSE) {
            ptx::mbar_arrive_expect_tx(&meta_full[ast], meta_tx);
            if (p.split) ptx::tma_load_5d(sEraw + ast * p.eraw_bytes, &tmE, &meta_full[ast], kb * 8, q0, 0, bg, p0);
            else ptx::tma_load_4d(sEraw + ast * p.eraw_bytes, &tmE, &meta_full[ast], kb * 8, q0, b0, p0);
          }
          if (p.split) ptx::tma_load_5d_pair(sA + ast * p.a_bytes, &tmA, &a_full[ast], kb * 64, q0, 0, bg, p0);
          else ptx::tma_load_4d_pair(sA + ast * p.a_bytes, &tmA, &a_full[ast], kb * 64, q0, b0, p0);
          if (++ast == p.a_stages) { ast = 0; aph ^= 1u; }
        }
      }
    }
  } else if (warp == 0) {
    // ------------------------------------------------------------ W taps (fused: the pruning warps fetch dL/dO themselves)
    if (ptx::elect_one()) {
      const uint32_t w_tx = 2u * (uint32_t)C::kTapBBytes;
      bool alive = true;
      int wst = 0;
      uint32_t wph = 0;
      for (int lt = 0; alive && lt < my_tiles; ++lt) {
        int n0, w0_unused, h0_unused, b0_unused, c;
        locate(lt, n0, w0_unused, h0_unused, b0_unused, c);
        const int kb0 = first_k_block(p, n0, C::kKB);
        n0 += n_half;
        const HaloClass cl = class_of(c);
        const int taps = cl.R * cl.sb;  // filter taps served by one A box
        for (int ku = 0; alive && ku < p.k_uses; ++ku) {
          const int kl = ku / p.ss, si = ku - kl * p.ss, kb = kb0 + kl;
          for (int t = 0; t < taps; ++t) {
            if (!ptx::mbar_wait<kIdleWaitNs>(&w_empty[wst], wph ^ 1u, err, 0x180u + wst)) { alive = false; break; }
            if (rank == 0) ptx::mbar_arrive_expect_tx(&w_ready[wst], w_tx);
            const int r = t / cl.sb, s = t - r * cl.sb + si;
            const int ft = (cl.r_first + p.r_step * r) * p.S_full + cl.s_first + p.s_step * s;
#pragma unroll
            for (int j = 0; j < C::kBoxes; ++j)
              ptx::tma_load_2d_pair(sW + wst * p.w_bytes + j * C::kBoxBytes, &tmB, &w_ready[wst],
                                    ft * p.Cin + n0 + C::kBoxCols * j, kb * C::kKB);
            if (++wst == WS) { wst = 0; wph ^= 1u; }
          }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------- MMA issuer (first CTA only)
    // The whole warp walks the loops together and one elected lane issues the tensor-core instructions: every
    // address and descriptor word is then the same in all lanes, which lets the compiler keep them in the warp's
    // uniform registers, where those instructions take their operands from. The path per tap is kept short: one
    // barrier wait, running descriptor words updated by additions, compile-time offsets for the strips and the four
    // MMAs of a channel block.
    if (rank == 0) {
      const bool leader = ptx::elect_one();
      const uint32_t tmem_base = __shfl_sync(0xFFFFFFFFu, tmem_base_any, 0);  // one value for the warp, and known to be
      const uint32_t idesc = make_idesc(BN, SPARSE) & ~(p.f16 ? kIdescBf16Operands : 0u);
      // descriptors as two 32-bit halves: the start address only ever changes the low word
      const uint64_t adesc0 = ptx::make_smem_desc(0, 16, (uint32_t)p.pitch * 128u, 2);
      const uint64_t bdesc0 = ptx::make_smem_desc(0, C::kBoxBytes, 8 * C::kRowB, C::kBSwizzle);
      // metadata window: 16 groups of 8 consecutive 16-byte lines, one pitch of lines apart
      const uint64_t edesc0 = ptx::make_smem_desc(0, 128, (uint32_t)p.pitch * 16u, 0);
      const uint32_t a_hi = (uint32_t)(adesc0 >> 32), b_hi = (uint32_t)(bdesc0 >> 32), e_hi = (uint32_t)(edesc0 >> 32);
      const uint32_t a_lo0 = (uint32_t)adesc0 + (ptx::smem_u32(sA) >> 4);
      const uint32_t b_lo0 = (uint32_t)bdesc0 + (ptx::smem_u32(sW) >> 4);
      const uint32_t e_lo0 = (uint32_t)edesc0 + (ptx::smem_u32(sMeta) >> 4);
      const uint32_t a_stage16 = (uint32_t)p.a_bytes >> 4, w_stage16 = (uint32_t)p.w_bytes >> 4,
                     e_stage16 = (uint32_t)p.meta_bytes >> 4, m1_off16 = (uint32_t)p.m0_bytes >> 4;
      // first line (16-byte units) of the window of vertical tap offset dr = R-1-r: master dr % 2, pair dr / 2
      auto meta_row16 = [&p, m1_off16](int dr) -> uint32_t {
        const int off = dr * p.tb;  // box rows
        return ((off & 1) ? m1_off16 : 0u) + (uint32_t)((off >> 1) * 2 * p.pitch);
      };
      constexpr uint32_t kBStep = (uint32_t)((C::kKB / 4) * C::kRowB / 16);  // W rows of one MMA
      constexpr uint32_t kSlotCols = 4u * NT;                                // metadata columns of one W stage
      bool alive = true;
      int ast = 0, acc = 0, wst = 0;
      uint32_t aph = 0, wph = 0, cph = 0;
      // running words of the W ring: W descriptor, metadata column (relative)
      uint32_t b_lo = b_lo0, mcol = 0;
      // (a wait that gives up in one lane ends the role for the whole warp)
      auto wait_all = [&](uint64_t* bar, uint32_t parity, unsigned int code) -> bool {
        return __all_sync(0xFFFFFFFFu, ptx::mbar_wait(bar, parity, err, code));
      };
      for (int lt = 0; alive && lt < my_tiles; ++lt) {
        if (!wait_all(&acc_empty[acc], cph ^ 1u, 0x200u + acc)) break;
        // shared metadata region: the first columns of the other tile set's accumulators,
        // which the epilogue of the previous tile set reads out first
        if (p.meta_shared && lt > 0 && !wait_all(&meta_free[acc ^ 1], (((uint32_t)lt - 1u) >> 1) & 1u, 0x800u + acc)) break;
        const uint32_t meta_base = tmem_base + (uint32_t)(p.meta_shared ? (acc ^ 1) * set_cols : p.meta_col);
        ptx::tc_fence_after_sync();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc * set_cols);
        int c;
        unit_of(lt, c);
        const HaloClass cl = class_of(c);
        const int taps = cl.R * cl.sb;
        const uint32_t a_first16 = (uint32_t)(((cl.R - 1) * p.tb * p.pitch + (cl.sb - 1)) * 8);  // tap (0,0), in 16-byte units
        const uint32_t a_rowstep16 = (uint32_t)((p.tb * p.pitch - (cl.sb - 1)) * 8);             // last tap of a filter row -> first of the next
        const uint32_t strips = strip_mask(lt);
        const bool all_strips = strips == ((1u << NT) - 1u);
        // (this warp's instructions are the MMAs' issue rate: one form for whole blocks, one for the rest, no division for whole ones)
        const bool partial = p.last_mmas != 4;
        int kb0 = 0;
        if (partial && p.diag_cin_g != 0) {
          int n0, w0, h0, b0;
          locate(lt, n0, w0, h0, b0, c);
          kb0 = first_k_block(p, n0, C::kKB);
        }
        uint32_t accumulate = 0u;
        for (int ku = 0; alive && ku < p.k_uses; ++ku) {
          if (!wait_all(&a_full[ast], aph, 0x300u + ast)) { alive = false; break; }
          if (SPARSE && !FUSED && !wait_all(&meta_ready[ast], aph, 0x340u + ast)) { alive = false; break; }
          const int mmas = (partial && kb0 + ku / p.ss == p.k_last) ? p.last_mmas : 4;
          uint32_t a_lo = a_lo0 + (uint32_t)ast * a_stage16 + a_first16;
          int s = cl.sb, dr = cl.R - 1;
          const uint32_t e_stage = e_lo0 + (uint32_t)ast * e_stage16;
          uint32_t e_lo = e_stage + meta_row16(dr) + (uint32_t)(cl.sb - 1);
          for (int t = 0; t < taps; ++t) {
            if (!wait_all(&w_ready[wst], wph, 0x380u + wst)) { alive = false; break; }
            ptx::tc_fence_after_sync();
            const uint32_t e_col = meta_base + mcol;  // even: slots are 4 columns apart
            // MMAS: MMAs of the channel block if every strip takes part (no per-strip test in the issue path), 0: neither is known. Whole and half
            // blocks have a form of their own: with 64 output channels, the tests of the last form are what a tap waits for. Us, prune kernel
            // included, half blocks through the last form and their own: 8 x 6 x 6 images, 192 -> 64 channels, 5 x 5, 11.4 -> 10.4; 22 x 7 x 7, 384 -> 64,
            // 8.0 -> 7.6; 64 x 28 x 28, 64 -> 64, fused, 16.9 -> 16.1. (Forms for one and three MMAs too made every form slower: 512 x 32 x 32, 64 -> 128,
            // 75 -> 84.)
            auto issue_tap = [&](auto mmas_tag) {
              constexpr int MMAS = decltype(mmas_tag)::value;
              if (SPARSE) {
#pragma unroll
                for (int j = 0; j < NT; ++j)
                  if (MMAS || (strips & (1u << j)))
                    ptx::tc_cp_128x128b_pair(e_col + 4u * j, ((uint64_t)e_hi << 32) | (e_lo + (uint32_t)(8 * j)));
              }
#pragma unroll
              for (int j = 0; j < NT; ++j) {
                if (!MMAS && !(strips & (1u << j))) continue;
#pragma unroll
                for (int q = 0; q < (MMAS ? MMAS : 4); ++q) {
                  if (!MMAS && q >= mmas) continue;  // (not break: 18 x 18, 224 channels in 7 groups, 5 x 5, 15.2 us, so 14.7)
                  // strip j: 8 pixels = 1024 bytes to the right; MMA q: 32 bytes along the row
                  const uint64_t a_q = ((uint64_t)a_hi << 32) | (a_lo + (uint32_t)(j * 64 + q * 2));
                  const uint64_t b_q = ((uint64_t)b_hi << 32) | (b_lo + (uint32_t)q * kBStep);
                  if (SPARSE)
                    ptx::mma_sp_f16_ss_pair(d_tmem + (uint32_t)(j * BN), a_q, b_q, e_col + (uint32_t)(4 * j + (q & 2)),
                                            idesc | (uint32_t)(q & 1), q == 0 ? accumulate : 1u);
                  else
                    ptx::mma_f16_ss_pair(d_tmem + (uint32_t)(j * BN), a_q, b_q, idesc, q == 0 ? accumulate : 1u);
                }
              }
            };
            if (leader) {
              if (all_strips && mmas == 4) issue_tap(std::integral_constant<int, 4>{});
              else if (all_strips && mmas == 2) issue_tap(std::integral_constant<int, 2>{});
              else issue_tap(std::integral_constant<int, 0>{});
              ptx::tc_commit_pair(&w_empty[wst], 3);
            }
            accumulate = 1u;
            // next tap: one pixel to the left, or the end of the filter row above
            if (--s == 0) { s = cl.sb; a_lo -= a_rowstep16; --dr; e_lo = e_stage + meta_row16(dr) + (uint32_t)(cl.sb - 1); }
            else { a_lo -= 8u; e_lo -= 1u; }
            if (++wst == WS) { wst = 0; wph ^= 1u; b_lo = b_lo0; mcol = 0; }
            else { b_lo += w_stage16; mcol += kSlotCols; }
          }
          if (alive && leader) ptx::tc_commit_pair(&a_empty[ast], 3);
          if (++ast == p.a_stages) { ast = 0; aph ^= 1u; }
        }
        if (alive && leader) ptx::tc_commit_pair(&acc_full[acc], 3);
        if (++acc == 2) { acc = 0; cph ^= 1u; }
      }
    }
  } else if (!FUSED && warp < 6) {
    // ------------------------------------------------- metadata rearranger (two-pass)
    // Once per A box the four warps turn the row-major metadata box TMA delivered into the two masters
    // (one 16-byte line per lane and pass: two 16-byte loads, four prmt, one 16-byte store), then arrive
    // on meta_ready. Every warp waits for every box in turn (a parity wait must see each phase).
    if (SPARSE) {
      const int mw = warp - 2;
      const int lines0 = p.pairs0 * 2 * p.pitch, lines = (p.pairs0 + p.pairs1) * 2 * p.pitch;
      const int a_uses = my_tiles * p.k_uses;
      constexpr int kBatch = 3;  // lines per lane whose loads are issued before any store
      for (int ause = 0; ause < a_uses; ++ause) {
        const int ast = ause & (p.a_stages - 1);
        if (!ptx::mbar_wait(&meta_full[ast], (uint32_t)(ause >> p.a_shift) & 1u, err, 0x500u + ast)) break;
        const uint8_t* raw = sEraw + ast * p.eraw_bytes;
        uint8_t* master = sMeta + ast * p.meta_bytes;
        for (int first = mw * 32 + lane; first < lines; first += 128 * kBatch) {
          uint4 lo[kBatch], hi[kBatch];
          uint32_t sel[kBatch];
#pragma unroll
          for (int k = 0; k < kBatch; ++k) {
            const int L = first + 128 * k;
            if (L < lines) {
              const int pi = L >= lines0 ? 1 : 0;
              const int l = L - pi * lines0;
              const int m2e = (int)(((uint32_t)l * p.pitch_magic) >> 20), x = l - m2e * p.pitch;  // 2m + e, pixel column
              const int row_a = (pi + (m2e & ~1)) * p.pitch + x;  // box pixel (pi + 2m, x); its partner is one box row down
              lo[k] = *(const uint4*)(raw + row_a * 16);
              hi[k] = *(const uint4*)(raw + (row_a + p.pitch) * 16);
              sel[k] = (m2e & 1) ? 0x7632u : 0x5410u;
            }
          }
#pragma unroll
          for (int k = 0; k < kBatch; ++k) {
            const int L = first + 128 * k;
            if (L < lines)
              *(uint4*)(master + L * 16) =
                  make_uint4(well_formed(prmt(lo[k].x, hi[k].x, sel[k])), well_formed(prmt(lo[k].y, hi[k].y, sel[k])),
                             well_formed(prmt(lo[k].z, hi[k].z, sel[k])), well_formed(prmt(lo[k].w, hi[k].w, sel[k])));
          }
        }
        ptx::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive_cluster(&meta_ready[ast], 0);
      }
    }
  } else if (FUSED && (((warp & 3) != 1 && (warp < 4 || warp >= 8)) || warp == 9 || warp == 13 || warp == 17 || warp == 21)) {
    // ------------------------------------------------------------ pruner
    // Work unit = 8 pixel rows of a box = one pass of a warp: lane = (row, c), and the thread owns vectors
    // c, c + 4, c + 8 and c + 12 (8 channels each) of the row's 16, so that every load instruction of the
    // warp reads 64 contiguous bytes per pixel. Units are numbered through all boxes of this CTA and dealt
    // round-robin to the pruning warps. A thread reads its 64 bytes of dense dL/dO straight from global
    // memory into registers (the loads of the next unit go out as soon as this one is pruned, and the lines
    // of the next box are asked into L2 a box ahead), prunes them and writes the compressed vectors and their
    // metadata into the A stage. These stores replace the TMA write of the compressed box, so the fused mode adds no
    // shared-memory traffic to the two-pass kernel's - which matters because with 64 or 128 input
    // channels the MMAs themselves are bound by shared-memory reads.
    {
      // number of this pruning warp, 0 .. kPruneWarps - 1: warps 2, 3, 8, then 10.. without those on scheduler 1 (0..13),
      // then the four on scheduler 1
      const int pw = warp == 9 ? 14 : warp == 13 ? 15 : warp == 17 ? 16 : warp == 21 ? 17 : warp < 4 ? warp - 2 : warp == 8 ? 2 : 3 + (warp - 10) - ((warp - 9) >> 2);
      const int upb = p.units_per_box;
      if (p.static_pad) {
        // every stage starts out as padding: zero values, metadata naming the position pair (0, 1)
        const int words = p.a_stages * p.a_bytes >> 4;
        for (int k = pw * 32 + lane; k < words; k += 32 * kPruneWarps) ((uint4*)sA)[k] = make_uint4(0u, 0u, 0u, 0u);
        const int mwords = p.a_stages * p.meta_bytes >> 4;
        for (int k = pw * 32 + lane; k < mwords; k += 32 * kPruneWarps)
          ((uint4*)sMeta)[k] = make_uint4(0x44444444u, 0x44444444u, 0x44444444u, 0x44444444u);
        ptx::fence_proxy_async_smem();
        ptx::named_bar_sync(3, 32 * kPruneWarps);  // no unit is announced before every stage is cleared
      }
      const int a_uses = my_tiles * p.k_uses;
      const int row8 = lane >> 2, c = lane & 3;
      const uint32_t px_bytes = (uint32_t)p.Cout * 2u;
      const int tb_shift = p.tb == 4 ? 2 : p.tb >> 1;  // tb is 1, 2 or 4
      auto prune_units = [&](auto m_tag, auto n_tag, auto scheme_tag) {
        constexpr int M = decltype(m_tag)::value;
        constexpr int N = decltype(n_tag)::value;
        constexpr int SCHEME = decltype(scheme_tag)::value;
        // ---- load cursor: the unit whose loads go out next, and the box it lies in
        int ia = 0, o = pw, lt = 0, ku = 0;  // ku: box of the tile set (channel block ku / ss, filter column ku % ss)
        auto normalise = [&]() { while (o >= upb) { o -= upb; ++ia; if (++ku == p.k_uses) { ku = 0; ++lt; } } };
        normalise();
        int org_box = -1;             // box the origin below belongs to
        const uint8_t* org_ptr = p.a_dense;  // address of box pixel (0, 0), channel block kb, quarter c (may lie outside the tensor)
        int org_p = 0, org_q = 0;     // dO pixel of box pixel (0, 0)
        int org_b = 0;                // its image
        int64_t org_pix = 0;          // its linear pixel number (random keys)
        bool org_ok = false;
        int org_kb0 = 0;              // first channel block of its tile's window
        auto set_origin = [&](int box_lt, int box_ku, const uint8_t*& ptr, int& p0, int& q0, int& b0, int64_t& pix, bool& ok, int& kb0) {
          int n0, w0, h0, parity;
          ok = locate(box_lt, n0, w0, h0, b0, parity);
          const int box_kl = box_ku / p.ss, si = box_ku - box_kl * p.ss;
          kb0 = first_k_block(p, n0, 128);
          const int box_kb = kb0 + box_kl;
          q0 = w0 + p.pad_w - (p.sb - 1) - si;
          p0 = h0 + p.pad_h - (p.R - 1);
          pix = ((int64_t)b0 * p.P + p0) * p.Q + q0;
          ptr = p.a_dense + pix * (int64_t)px_bytes + box_kb * 256 + c * 16;
        };
        // box pixel (box row br, column col) -> image offset, pixel row and pixel column relative to the origin
        auto box_pixel = [&](int br, int col, int& ib, int& ih, int& iw) {
          ih = br >> tb_shift;
          ib = (br & (p.tb - 1)) * p.img_per_row;
          iw = col;
          if (p.split) { ib += col >> 2; iw = col & 3; }
        };
        // The unit whose loads are in flight: its 64 bytes, its pixel row in the box, its box
        uint4 w[4];
        int u_i = 0, u_ia = 0, u_kb = 0;  // (u_kb: channel block)
        int64_t u_pix = 0;
        bool u_live = false;  // some pixel of the unit lies inside the tensor (halo rows above / below an image: none does)
        auto fetch = [&]() {
          if (org_box != ia) {
            set_origin(lt, ku, org_ptr, org_p, org_q, org_b, org_pix, org_ok, org_kb0);
            org_box = ia;
            // ask the lines of the NEXT box into L2 now, a whole box ahead of their loads: 2 lines of 128
            // bytes per box pixel, dealt to the pruning threads
            int nlt = lt, nkb = ku + 1;
            if (nkb == p.k_uses) { nkb = 0; ++nlt; }
            if (ia + 1 < a_uses) {
              const uint8_t* nptr;
              int np0, nq0, nb0, nkb0;
              int64_t npix;
              bool nok;
              set_origin(nlt, nkb, nptr, np0, nq0, nb0, npix, nok, nkb0);
              for (int line = pw * 32 + lane; line < 2 * p.img_rows; line += 32 * kPruneWarps) {
                const int px = line >> 1;
                const int br = (int)(((uint32_t)px * p.pitch_magic) >> 20);  // box row
                int ib, ih, iw;
                box_pixel(br, px - br * p.pitch, ib, ih, iw);
                if (nok && nb0 + ib < p.B && (unsigned)(np0 + ih) < (unsigned)p.P && (unsigned)(nq0 + iw) < (unsigned)p.Q)
                  asm volatile("prefetch.global.L2 [%0];" ::"l"(nptr - c * 16 + (uint32_t)((ib * p.P + ih) * p.Q + iw) * px_bytes + (line & 1) * 128));
              }
            }
          }
          if (p.static_pad) {
            const int ur = NT == 2 ? (o >> 1) : o, uc = NT == 2 ? (o & 1) : 0;
            u_i = (p.unit_row0 + ur) * p.pitch + p.unit_col0 + 8 * uc + row8;
          } else {
            u_i = 8 * o + row8;
          }
          u_ia = ia;
          const int kb = org_kb0 + ku / p.ss;
          u_kb = kb;
          const int br = (int)(((uint32_t)u_i * p.pitch_magic) >> 20);  // box row
          int ib, ih, iw;
          box_pixel(br, u_i - br * p.pitch, ib, ih, iw);
          const uint32_t off = (uint32_t)((ib * p.P + ih) * p.Q + iw);
          u_pix = org_pix + off;
          const bool valid = org_ok && u_i < p.img_rows && org_b + ib < p.B && (unsigned)(org_p + ih) < (unsigned)p.P &&
                             (unsigned)(org_q + iw) < (unsigned)p.Q;
          u_live = __any_sync(0xFFFFFFFFu, valid);
#pragma unroll
          for (int v = 0; v < 4; ++v) w[v] = make_uint4(0u, 0u, 0u, 0u);
          if (valid) {
            const uint8_t* src = org_ptr + off * px_bytes;
            // vector c + 4v: channels beyond Cout (a last channel block that is half empty) read as zero
            const int chan0 = kb * 128 + c * 8;
#pragma unroll
            for (int v = 0; v < 4; ++v)
              if (chan0 + 32 * v < p.Cout) w[v] = ldg_stream(src + 64 * v);
          }
          o += kPruneWarps;
          normalise();
        };
        int boxes_seen = 0;  // stage hand-backs (a_empty phases) this warp has observed, one per box, in order
        int pending_ast = -1;  // stage of the unit whose stores are out but not yet announced
        // Makes the stores of the previous unit visible to the tensor core and announces them. Called a whole
        // unit later than the stores were issued, so the fence finds them done.
        auto announce = [&]() {
          if (pending_ast >= 0) {
            ptx::fence_proxy_async_smem();  // the tensor core reads A and the masters through the async proxy
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_cluster(&a_full[pending_ast], 0);
          }
        };
        bool more = ia < a_uses;  // a unit is in flight
        if (more) fetch();
        while (more) {
          const int i = u_i, cia = u_ia;
          const bool live = u_live;
          const int ast = cia & (p.a_stages - 1);
          uint2 out[4];
          uint32_t metaw;
          // (a group of M channels = vectors c + 4v of M / 8 neighbouring lanes c, same v)
          if (live) {
            fused_prune_vectors<M, N, SCHEME, false>(w, u_pix * (p.Cout >> 3) + u_kb * 16 + c, 4, p.seed_lo, p.seed_hi, c & (M / 8 - 1), out, metaw);
          } else {
            // a unit of padding only: zeros, whatever positions the metadata names (it names the pair (0, 1))
#pragma unroll
            for (int v = 0; v < 4; ++v) out[v] = make_uint2(0u, 0u);
            metaw = 0x44444444u;
          }
          // the registers of this unit are free: the loads of the next one go out before this one's stores
          more = ia < a_uses;
          if (more) fetch();
          // only now, with the unit pruned and the next one's loads in flight, does the warp need the stage
          if (boxes_seen <= cia) {  // the MMAs that read this stage's previous contents (box cia - 2) have completed
            // (whatever this warp still owes an earlier box goes out first: with fewer units per box than pruning warps
            // the stage waited for here can be the very one that unit belongs to)
            announce();
            pending_ast = -1;
            bool ok = true;
            while (boxes_seen <= cia) {
              const int bs = boxes_seen & (p.a_stages - 1);
              if (!ptx::mbar_wait<kIdleWaitNs>(&a_empty[bs], (((uint32_t)boxes_seen >> p.a_shift) & 1u) ^ 1u, err, 0x900u + bs)) { ok = false; break; }
              ++boxes_seen;
            }
            if (!__all_sync(0xFFFFFFFFu, ok)) break;
          }
          announce();
          const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, metaw, 1);  // (all lanes: before the rows part ways)
          if (i < p.img_rows) {
            const int sw = i & 7;
            // vector j = c + 4v -> 8 bytes at 16-byte chunk j / 2 = 2v + c / 2 (swizzled), half j % 2 = c % 2
            uint8_t* a_row = sA + ast * p.a_bytes + i * 128 + 8 * (c & 1);
            const int ch0 = (c >> 1) ^ sw;
#pragma unroll
            for (int v = 0; v < 4; ++v) *(uint2*)(a_row + ((ch0 ^ (2 * v)) << 4)) = out[v];
            // Metadata: byte v of metaw belongs to the 16-channel group 2v + c / 2, i.e. to 32-bit word v of the
            // master line e = c / 2, byte c % 2 of its low or high half-word. Lanes c and c ^ 1 hold the two bytes
            // of each half-word: they trade words, the even lane writes the half-words of v = 0, 1, the odd one
            // those of v = 2, 3.
            const uint32_t lo = (c & 1) ? other : metaw, hi = (c & 1) ? metaw : other;  // bytes of c even / c odd
            const uint32_t pair = (c & 1) ? prmt(lo, hi, 0x7362) : prmt(lo, hi, 0x5140);  // two half-words
            const int ih = (int)(((uint32_t)i * p.pitch_magic) >> 20), iw = i - ih * p.pitch;  // ih: box row
            uint8_t* master = sMeta + ast * p.meta_bytes + (iw << 4) + 8 * (c & 1) + (c >> 1) * (p.pitch << 4);
            if (ih < 2 * p.pairs0) {
              uint8_t* dst = master + (((ih & ~1) * p.pitch) << 4) + 2 * (ih & 1);
              *(uint16_t*)dst = (uint16_t)pair;
              *(uint16_t*)(dst + 4) = (uint16_t)(pair >> 16);
            }
            if (ih >= 1 && ih <= 2 * p.pairs1) {
              uint8_t* dst = master + p.m0_bytes + ((((ih - 1) & ~1) * p.pitch) << 4) + 2 * ((ih - 1) & 1);
              *(uint16_t*)dst = (uint16_t)pair;
              *(uint16_t*)(dst + 4) = (uint16_t)(pair >> 16);
            }
          }
          pending_ast = ast;
        }
        announce();
      };
      using std::integral_constant;
      auto with_m = [&](auto m_tag) {
        if (p.fused_scheme == SDGP_MAGNITUDE) {
          if (p.fused_n == 1) prune_units(m_tag, integral_constant<int, 1>{}, integral_constant<int, SDGP_MAGNITUDE>{});
          else prune_units(m_tag, integral_constant<int, 2>{}, integral_constant<int, SDGP_MAGNITUDE>{});
        } else if (p.fused_scheme == SDGP_RANDOM) {
          if (p.fused_n == 1) prune_units(m_tag, integral_constant<int, 1>{}, integral_constant<int, SDGP_RANDOM>{});
          else prune_units(m_tag, integral_constant<int, 2>{}, integral_constant<int, SDGP_RANDOM>{});
        } else {
          if (p.fused_n == 1) prune_units(m_tag, integral_constant<int, 1>{}, integral_constant<int, SDGP_RESCALED_MAGNITUDE>{});
          else prune_units(m_tag, integral_constant<int, 2>{}, integral_constant<int, SDGP_RESCALED_MAGNITUDE>{});
        }
      };
      if (p.fused_m == 4) with_m(integral_constant<int, 4>{});
      else if (p.fused_m == 8) with_m(integral_constant<int, 8>{});
      else if (p.fused_m == 16) with_m(integral_constant<int, 16>{});
      else with_m(integral_constant<int, 32>{});
    }
  } else if (warp >= kEpilogueWarp0 && warp < kEpilogueWarp0 + 4) {
    // ------------------------------------------------------------ epilogue
    const int q = warp & 3;
    const int row = q * 32 + lane;
    // this thread's pixel of a strip: strip row row / 8 = (pixel row, image), 8 pixels to a row (column-split mode: 4 pixels
    // of two neighbouring images)
    const int srow = row >> 3, dh = srow / p.tb, px = row & 7;
    const int db = (srow % p.tb) * p.img_per_row + (p.split ? px >> 2 : 0), dw = p.split ? px & 3 : px;
    uint32_t cph = 0, chunk = 0;
    int acc = 0;
    for (int lt = 0; lt < my_tiles; ++lt) {
      int n0, w0, h0, b0, c;
      const bool in_range = locate(lt, n0, w0, h0, b0, c);
      const uint32_t strips = strip_mask(lt);
      // (patches: the four warps stay or leave together, they meet at a named barrier in every slab)
      const bool ready = ptx::mbar_wait<kIdleWaitNs>(&acc_full[acc], cph, err, 0x600u + acc);
      if (PATCH ? !ptx::named_bar_all(1, 128, ready) : !ready) break;
      ptx::tc_fence_after_sync();
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * set_cols + j * BN);
        uint64_t* first_slab_read = (p.meta_shared && j == 0) ? &meta_free[acc] : nullptr;
        uint64_t* released = j == NT - 1 ? &acc_empty[acc] : nullptr;
        const bool strip_live = in_range && (strips & (1u << j));
        if constexpr (FUSED) {
          // this warp's 4 strip rows: 4 / tb pixel rows of tb images
          const int hq = h0 + q * (4 / p.tb);
          if (p.split) store_box<BN>(taddr, sOut + q * p.out_bufs * kSlabBytes, &tmD.m[0], true, n0, 0, 2 * j, b0 / p.img_per_row, hq, strip_live,
                                     p.d.channels - n0, first_slab_read, released, p.f16 != 0, p.out_bufs, chunk);
          else store_box<BN>(taddr, sOut + q * p.out_bufs * kSlabBytes, &tmD.m[0], false, n0, w0 + 8 * j, b0, hq, 0, strip_live && w0 + 8 * j < p.W,
                             p.d.channels - n0, first_slab_read, released, p.f16 != 0, p.out_bufs, chunk);
        } else if constexpr (PATCH) {
          if (p.split) store_patch<BN, true>(taddr, sOut, p.out_bufs, &tmD.m[0], n0, 0, 2 * j, b0 / p.img_per_row, h0, strip_live, chunk,
                                             first_slab_read, p.f16 != 0);
          else store_patch<BN, false>(taddr, sOut, p.out_bufs, &tmD.m[c], n0, w0 + 8 * j, b0, h0, 0,
                                      strip_live && w0 + 8 * j < p.cls[c].W && h0 < p.cls[c].H, chunk, first_slab_read, p.f16 != 0);
          if (released != nullptr) {
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_cluster(released, 0);
          }
        } else {
          const int w = w0 + dw + (p.split ? 0 : 8 * j), h = h0 + dh, b = b0 + db + (p.split ? 2 * j : 0);
          const bool inside = strip_live && w < p.W && h < p.H && b < p.B;
          uint8_t* dst = inside ? p.d.base + b * p.d.sb + h * p.d.sh + w * p.d.sw + 2 * n0 : nullptr;
          store_rows<BN>(taddr, dst, p.d.channels - n0, p.d.aligned32 != 0, first_slab_read, released, p.f16 != 0);
        }
      }
      if (++acc == 2) { acc = 0; cph ^= 1u; }
    }
    // the staging rows have been read; the writes themselves complete with the grid (whoever depends on dD waits for that)
    if ((FUSED || PATCH) && lane == 0) ptx::bulk_wait_group_read<0>();
  }

  __syncwarp();
  if (*(volatile unsigned int*)err != 0u) {
    const uint64_t t0 = ptx::globaltimer_ns();
    while (ptx::globaltimer_ns() - t0 < 200000ull) {
    }
  }
  ptx::tc_fence_before_sync();
  __syncwarp();
  ptx::cluster_sync();
  ptx::tc_fence_after_sync();
  if (warp == 1) ptx::tmem_dealloc_pair(tmem_base, kTmemCols);
}

// Shared-memory and TMEM plan of the whole-filter-reuse kernel. Returns false if it does not fit.
template <bool SPARSE, int BN, bool FUSED>
bool plan_halo(HaloParams* p, int nt) {
  using C = Cfg<SPARSE, BN>;
  const int budget = kSmemLimit - kSmemSlack;
  {
    if (nt * BN > 256) return false;         // two tile sets of accumulators must fit the 512 TMEM columns
    p->split = (p->W == 4) ? 1 : 0;  // images 4 pixels wide: two per strip row, horizontal taps by separate boxes
    if (!p->split && nt == 2 && p->W <= 8) return false;  // a second strip would be empty
    p->nt = nt;
    p->img_per_row = p->split ? 2 * nt : 1;
    if (p->B % p->img_per_row != 0) return false;  // a box row of images must not reach past the batch
    p->ss = p->split ? p->S : 1;
    p->sb = p->split ? 1 : p->S;
    p->k_uses = p->k_blocks * p->ss;
    p->pitch = 8 * nt + p->sb - 1;
    p->th = p->H <= 4 ? 4 : p->H <= 8 ? 8 : kHaloRows;
    p->tb = kHaloRows / p->th;
    p->img_h = (p->th + p->R - 1) * p->tb;
    p->img_rows = p->pitch * p->img_h;
    p->static_pad = 0;
    p->units_per_box = (p->img_rows + 7) / 8;
    if (p->pitch > 256 || p->img_h > 256) return false;
    if (p->classes == 4 && p->split) return false;
    p->a_bytes = round_up(p->img_rows * 128, 1024);
    p->eraw_bytes = (SPARSE && !FUSED) ? round_up(p->img_rows * 16, 128) : 0;
    p->w_bytes = C::kTapBBytes;
    // vertical tap offset dr = 0 .. R-1 starts tb * dr box rows down: master (tb * dr) % 2, pair (tb * dr) / 2
    p->pairs0 = 8 + (p->tb == 1 ? (p->R - 1) >> 1 : (p->tb >> 1) * (p->R - 1));
    p->pairs1 = (p->tb == 1 && p->R > 1) ? 8 + ((p->R - 2) >> 1) : 0;
    p->m0_bytes = SPARSE ? p->pairs0 * 2 * p->pitch * 16 : 0;
    p->meta_bytes = SPARSE ? round_up((p->pairs0 + p->pairs1) * 2 * p->pitch * 16, 128) : 0;
    p->sets_w = p->split ? 1 : (p->W + 8 * nt - 1) / (8 * nt);
    p->tiles_h = (p->H + p->th - 1) / p->th;
    const int tile_imgs = p->tb * p->img_per_row;  // images of one tile set
    const int64_t m_sets = (int64_t)p->sets_w * p->tiles_h * ((p->B + tile_imgs - 1) / tile_imgs);
    if (m_sets * p->tiles_n * p->classes > 0x3FFFFFFF) return false;
    p->m_sets = (int)m_sets;
    p->pair_tiles = (int)((m_sets + 1) / 2) * p->tiles_n * p->classes;
    // Stride 2 stores boxes: its classes have few taps, so that the stores set the pace, and dD's pixels are not neighbours. 128 -> 128
    // channels, 3 x 3 stride 2 at 56 x 56, batch 256: 2.29 M write requests at L2 a class as rows, 0.60 M as boxes; the four classes 89 us
    // -> 83. Stride 1 keeps the rows (128 -> 64 channels at 32 x 32, batch 512, prune kernel included: 82 us, as boxes 88).
    p->patch_store = (!FUSED && p->r_step == 2) ? 1 : 0;
    // A ring: two stages; four where a box feeds few taps (column-split mode: R taps per box), so that the loads
    // run further ahead of the MMAs, if that still leaves three W stages
    p->a_stages = 2;
    const int per_a = p->a_bytes + p->eraw_bytes + p->meta_bytes;
    if (p->split && (budget - 4 * per_a - 1024 - ((FUSED || p->patch_store) ? 4 * kSlabBytes : 0)) / p->w_bytes >= 3) p->a_stages = 4;
    p->a_shift = p->a_stages == 4 ? 2 : 1;
    const int fixed = p->a_stages * per_a + 1024;
    p->out_bufs = (FUSED || p->patch_store) ? 2 : 0;  // epilogue staging
    int w_stages = (budget - fixed - 4 * p->out_bufs * kSlabBytes) / p->w_bytes;
    if (p->out_bufs == 2 && w_stages < 4) {
      p->out_bufs = 1;
      w_stages = (budget - fixed - 4 * kSlabBytes) / p->w_bytes;
    }
    if (p->patch_store && w_stages < 3) {
      if (p->classes == 4) return false;
      p->patch_store = p->out_bufs = 0;
      w_stages = (budget - fixed) / p->w_bytes;
    }
    if (w_stages > kMaxStages) w_stages = kMaxStages;
    p->meta_shared = 0;
    p->meta_col = 2 * nt * BN;
    if (SPARSE) {
      const int slot_cols = 4 * nt;  // TMEM columns of one W stage's metadata
      const int free_cols = (int)kTmemCols - 2 * nt * BN;
      if (free_cols >= 3 * slot_cols) {
        if (w_stages > free_cols / slot_cols) w_stages = free_cols / slot_cols;
      } else {
        p->meta_shared = 1;  // slots live in the first 64 columns of the tile set being read out
        p->meta_col = 0;
        if (w_stages > 64 / slot_cols) w_stages = 64 / slot_cols;
      }
    }
    if (w_stages < 3) return false;
    p->w_stages = w_stages;
    p->off_eraw = p->a_stages * p->a_bytes;
    p->off_meta = p->off_eraw + p->a_stages * p->eraw_bytes;
    p->off_w = round_up(p->off_meta + p->a_stages * p->meta_bytes, 1024);
    p->pitch_magic = ((1u << 20) + (uint32_t)p->pitch - 1u) / (uint32_t)p->pitch;
    p->off_out = round_up(p->off_w + w_stages * p->w_bytes, 1024);
    p->off_bar = p->off_out + 4 * p->out_bufs * kSlabBytes;
    p->smem_bytes = p->off_bar + 512 + 1024;
    if (p->smem_bytes > kSmemLimit) return false;
    if (FUSED && p->sets_w == 1 && p->tiles_h == 1 && p->a_bytes % 16 == 0 && p->meta_bytes % 16 == 0) {
      // Box pixel row 0 is dL/dO row p0 and box column 0 is dL/dO column q0 (every tile set starts at h0 = w0 = 0); the
      // rows and columns of the box that lie inside dL/dO's P x Q pixels are the same for every box.
      const int p0 = p->pad_h - (p->R - 1), q0 = p->pad_w - (p->sb - 1);
      const int row_lo = p0 < 0 ? -p0 : 0;
      const int row_hi = (p->th + p->R - 1) < (p->P - p0) ? (p->th + p->R - 1) : (p->P - p0);
      const int col_lo = p->split ? 0 : (q0 < 0 ? -q0 : 0);
      const bool cols_fit = p->split ? p->Q <= 4 : (p->Q - q0 <= col_lo + 8 * nt);
      if (row_hi > row_lo && cols_fit) {
        p->static_pad = 1;
        p->unit_row0 = row_lo * p->tb;
        p->unit_col0 = col_lo;
        p->units_per_box = (row_hi - row_lo) * p->tb * nt;
      }
    }
    p->mg_tiles_n = div_magic((uint32_t)p->tiles_n);
    p->mg_sets_w = div_magic((uint32_t)p->sets_w);
    p->mg_tiles_h = div_magic((uint32_t)p->tiles_h);
    // The pair tiles of a last round that fills at most half the CTA pairs are dealt out strip by
    // strip: that round then costs about half.
    p->units = p->pair_tiles;
    p->split_from = p->pair_tiles;
    const int max_pairs = sm_count() / 2;
    const int rem = p->pair_tiles % max_pairs;
    if (nt == 2 && p->pair_tiles > max_pairs && rem > 0 && 2 * rem <= max_pairs) {
      p->split_from = p->pair_tiles - rem;
      p->units = p->pair_tiles + rem;
    }
    return true;
  }
  return false;
}

template <bool SPARSE, int BN, int NT, bool FUSED>
sdgp_status launch_halo_nt(const void* A, const void* meta, const void* Wt, const DgradView& view, HaloParams p,
                           cudaStream_t stream) {
  using C = Cfg<SPARSE, BN>;
  if (!plan_halo<SPARSE, BN, FUSED>(&p, NT)) return SDGP_ERR_UNSUPPORTED;

  if (p.classes == 1) p.cls[0] = HaloClass{p.R, p.S, p.sb, p.pad_h, p.pad_w, p.r_first, p.s_first, p.H, p.W};
  else
    for (HaloClass& c : p.cls) c.sb = c.S;
  CUtensorMap tmA, tmE, tmB;
  HaloOutMaps<true> tmD;
  p.d = view.d;
  p.early = early_for(SPARSE && !FUSED && p.last_launch, pairs_for(p.units));
  const int P = view.P, Q = view.Q;
  const uint64_t CA = (SPARSE && !FUSED) ? (uint64_t)view.a_channels / 2 : (uint64_t)view.a_channels;
  // Dimensions: channel, pixel column, [column-split mode only: image within a box row (img_per_row images lie side by
  // side),] image (group), pixel row. A box then holds its rows in (pixel row, image group) order and, inside a row,
  // image after image.
  const uint64_t ipr = (uint64_t)p.img_per_row, groups = (uint64_t)view.batch / ipr;
  const uint32_t box_w = (uint32_t)(p.split ? 4 : p.pitch), box_h = (uint32_t)(p.img_h / p.tb);
  // builds the map of a [B, rows, cols, chan] tensor of 2-byte elements with the given strides and box extents
  auto encode_nhwc = [&](CUtensorMap* tm, CUtensorMapDataType dt, const void* base, uint64_t chan, uint64_t cols, uint64_t rows,
                         uint64_t images, uint64_t s_col, uint64_t s_row, uint64_t s_img, uint32_t b_chan, uint32_t b_col,
                         uint32_t b_ipr, uint32_t b_grp, uint32_t b_row, CUtensorMapSwizzle swz) -> bool {
    if (p.split) {
      const uint64_t dims[5] = {chan, cols, ipr, images / ipr, rows};
      const uint64_t strides[4] = {s_col, s_img, s_img * ipr, s_row};
      const uint32_t box[5] = {b_chan, b_col, b_ipr, b_grp, b_row};
      return encode(tm, dt, 5, base, dims, strides, box, swz);
    }
    const uint64_t dims[4] = {chan, cols, images, rows};
    const uint64_t strides[3] = {s_col, s_img, s_row};
    const uint32_t box[4] = {b_chan, b_col, b_grp, b_row};
    return encode(tm, dt, 4, base, dims, strides, box, swz);
  };
  // (fused: the pruning warps read dL/dO with plain loads and the A map goes unused)
  if (!encode_nhwc(&tmA, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, A, CA, (uint64_t)Q, (uint64_t)P, (uint64_t)view.batch, CA * 2, CA * 2 * Q,
                   CA * 2 * Q * P, 64, box_w, (uint32_t)ipr, (uint32_t)p.tb, box_h, CU_TENSOR_MAP_SWIZZLE_128B))
    return SDGP_ERR_CUDA;
  tmE = tmA;
  p.a_dense = (const uint8_t*)A;
  if (SPARSE && !FUSED) {
    const uint64_t CE = (uint64_t)view.meta_channels / 16;
    if (!encode_nhwc(&tmE, CU_TENSOR_MAP_DATA_TYPE_UINT16, meta, CE, (uint64_t)Q, (uint64_t)P, (uint64_t)view.batch, CE * 2, CE * 2 * Q,
                     CE * 2 * Q * P, 8, box_w, (uint32_t)ipr, (uint32_t)p.tb, box_h, CU_TENSOR_MAP_SWIZZLE_NONE))
      return SDGP_ERR_CUDA;
  }
  {
    const uint64_t dims[2] = {(uint64_t)view.w_cols, (uint64_t)p.Cout};
    const uint64_t strides[1] = {(uint64_t)view.w_cols * 2};
    const uint32_t box[2] = {(uint32_t)C::kBoxCols, (uint32_t)C::kKB};
    if (!encode(&tmB, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Wt, dims, strides, box,
                C::kRowB == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B))
      return SDGP_ERR_CUDA;
  }
  tmD.m[0] = tmA;
  if (FUSED || p.patch_store) {
    // dD, a strip (fused: one warp's quarter of it) per store: 8 pixel columns (column-split mode: the 4 columns of two neighbouring images)
    for (int c = 0; c < p.classes; ++c) {
      const uint8_t* base = view.d.base;  // of parity (0, 0); a pixel of dD is half a step of the parities' images
      if (p.classes == 4) base += (c >> 1) * (view.d.sh / 2) + (c & 1) * (view.d.sw / 2);
      if (!encode_nhwc(&tmD.m[c], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, base, (uint64_t)view.d.channels, (uint64_t)p.cls[c].W, (uint64_t)p.cls[c].H,
                       (uint64_t)p.B, (uint64_t)view.d.sw, (uint64_t)view.d.sh, (uint64_t)view.d.sb, 64, (uint32_t)(p.split ? 4 : 8), 2,
                       (uint32_t)p.tb, (uint32_t)(FUSED ? 4 / p.tb : p.th), CU_TENSOR_MAP_SWIZZLE_128B))
        return SDGP_ERR_CUDA;
    }
  }
  for (int c = p.classes; c < 4; ++c) tmD.m[c] = tmD.m[0];
  auto launch = [&](auto patch_tag) -> sdgp_status {
    constexpr bool PATCH = decltype(patch_tag)::value;
    static bool configured[kMaxDevices] = {};
    auto kernel = dgrad_halo_kernel<SPARSE, BN, NT, FUSED, PATCH>;
    if (!configure_once(kernel, configured)) return SDGP_ERR_CUDA;
    HaloOutMaps<PATCH> maps;
    for (int c = 0; c < (PATCH ? 4 : 1); ++c) maps.m[c] = tmD.m[c];
    return launch_pairs(kernel, pairs_for(p.units), FUSED ? kThreadsHaloFused : kThreadsHalo, p.smem_bytes, stream, tmA, tmE, tmB, maps, p);
  };
  if constexpr (!FUSED)
    if (p.patch_store) return launch(std::true_type{});
  return launch(std::false_type{});
}

template <bool SPARSE, bool FUSED>
sdgp_status launch_halo(int bn, int nt, const void* A, const void* meta, const void* Wt, const DgradView& view, const HaloParams& p,
                        cudaStream_t stream) {
  switch (bn * nt) {
    case 64: return launch_halo_nt<SPARSE, 64, 1, FUSED>(A, meta, Wt, view, p, stream);
    case 128: return nt == 2 ? launch_halo_nt<SPARSE, 64, 2, FUSED>(A, meta, Wt, view, p, stream)
                             : launch_halo_nt<SPARSE, 128, 1, FUSED>(A, meta, Wt, view, p, stream);
    case 192: return launch_halo_nt<SPARSE, 192, 1, FUSED>(A, meta, Wt, view, p, stream);
    case 256: return nt == 2 ? launch_halo_nt<SPARSE, 128, 2, FUSED>(A, meta, Wt, view, p, stream)
                             : launch_halo_nt<SPARSE, 256, 1, FUSED>(A, meta, Wt, view, p, stream);
    default: return SDGP_ERR_UNSUPPORTED;
  }
}

template <bool SPARSE>
bool plan_halo_shape(int bn, int nt, HaloParams* p) {
  if (nt < 1 || nt > 2) return false;
  switch (bn) {
    case 64: return plan_halo<SPARSE, 64, false>(p, nt);
    case 128: return plan_halo<SPARSE, 128, false>(p, nt);
    case 192: return plan_halo<SPARSE, 192, false>(p, nt);
    case 256: return plan_halo<SPARSE, 256, false>(p, nt);
    default: return false;
  }
}

}  // namespace
}  // namespace sdgp
