// Data-gradient contraction dD = dOp . W on the sm_100a tensor cores (Section 2.1, Fig. 2/3).
//
// One persistent, warp-specialised kernel serves the fully connected layer and the stride-1
// convolution (an implicit GEMM whose K axis covers filter taps x output channels; a 4-element
// pruning chunk never straddles two taps), with A either dense dL/dO (tcgen05.mma) or
// 2:4-compressed dL/dO plus position metadata (tcgen05.mma.sp).
//
// CTA pairs (cta_group::2): the two CTAs of a cluster own two neighbouring 128-pixel patches
// and one BN-wide block of input channels. Each CTA stages its own A patch (+ metadata) and
// HALF of the W columns; one thread of the pair's first CTA issues 256-row MMAs that read
// both halves. What limits this kernel is the bytes an SM can pull in from L2 (about 64 B per
// clock), so everything is arranged to reuse what is already in shared memory:
//   * W column halves: half the W bytes per CTA and half the shared-memory reads of B;
//   * filter-row reuse: for an R x S filter one A "image" of TH + R - 1 pixel rows serves all R
//     vertical taps - a tap is just a row offset (a multiple of 8 rows, i.e. of the 1024-byte
//     swizzle period) in the A descriptor - so A is fetched S times instead of R*S times;
//   * resident W: when the layer's whole W slice fits next to two A stages it is loaded once
//     per CTA and never streamed again.
//
// Warp roles
//   warp 0      TMA producer (both CTAs): per stage one 4-D box of A (pixels outside the image
//               arrive as zeros), the matching box of metadata, and the W boxes of its half.
//   warp 1      MMA issuer (first CTA only): tcgen05.cp of the stage's metadata into TMEM,
//               four MMAs per (tap, channel block), tcgen05.commit to the stage's "empty" barrier.
//   warps 2-5   (sparse only) build the stage's metadata images: from the row-major order TMA
//               delivers to the lane/column order the tensor core reads from TMEM. Each warp
//               owns every fourth stage; with fused pruning these four warps and eight helper
//               warps (10-17) first prune the stage's pixel rows together.
//   warps 6-9   epilogue: TMEM -> registers -> bf16 -> global memory, overlapped with the next tile's
//               main loop through a second accumulator.
//
// Barriers: full / acc_empty / w_full are waited on by the first CTA only and collect arrivals
// from both (full: the producer's byte count plus the metadata warps' arrivals, so the MMA
// thread waits once per stage); empty / acc_full exist in both CTAs and are signalled together
// by a multicast tcgen05.commit; meta_full is local (each CTA's own metadata box).
// Every wait is bounded: a wait that runs out records a code in g_device_error, the role
// stops issuing work, every other wait then gives up at once, and the kernel frees its TMEM
// and returns.
#include "dgrad_general.cuh"

namespace sdgp {
namespace {

// Tiles per CTA pair from which the epilogue stores boxes (plan()): 1024 -> 256 channels at 14 x 14, batch 256, 3.5 tiles a pair:
// 37.8 us against 39.6 with rows; 256 -> 64 at 56 x 56: 154 against 164.
constexpr int kBoxStoreRounds = 2;
// Fused pruning in the general kernel: eight more warps (10..17) prune beside warps 2..5. A lone warp
// runs the pruning code at a quarter of an instruction per clock; twelve of them keep up with the
// rate at which a memory-bound layer's dense dL/dO arrives.
constexpr int kFusedHelperWarps = 8;
constexpr int kThreadsGemmFused = kThreadsGemm + 32 * kFusedHelperWarps;
constexpr int kFusedPruners = 128 + 32 * kFusedHelperWarps;

// Metadata of an A tile: from the row-major order TMA delivers (16 bytes per pixel row: one uint16
// per 16 channels of a 128-channel block) to the order tcgen05.cp moves into TMEM. For the MMA
// covering channels [32*k2, 32*k2+32) of the block the tensor core reads one 32-bit TMEM column:
// lane (row%8) + 8*half + 16*(row/16) holds in its low 16 bits the four position nibbles of
// channels 32*k2 + 16*half + [0,16) of the row with bit 3 clear, in its high 16 bits those of
// row + 8. One call builds the 16 bytes of TMEM lane `tl` from its two rows. Rows that carry no
// data (past the patch, or outside the image where TMA filled zeros) get the well-formed
// position pair (0,1) in every chunk.
__device__ __forceinline__ void build_metadata_lane(const uint8_t* raw_rows, uint8_t* hw_tile, int tl, int rows_used) {
  const int row_a = ((tl >> 4) << 4) + (tl & 7), row_b = row_a + 8;
  const uint32_t sel = (tl & 8) ? 0x7632u : 0x5410u;
  const uint4 k01 = make_uint4(0x44444444u, 0x44444444u, 0x44444444u, 0x44444444u);
  uint4 lo = k01, hi = k01;
  if (row_a < rows_used) lo = *(const uint4*)(raw_rows + row_a * 16);
  if (row_b < rows_used) hi = *(const uint4*)(raw_rows + row_b * 16);
  *(uint4*)(hw_tile + tl * 16) =
      make_uint4(well_formed(prmt(lo.x, hi.x, sel)), well_formed(prmt(lo.y, hi.y, sel)),
                 well_formed(prmt(lo.z, hi.z, sel)), well_formed(prmt(lo.w, hi.w, sel)));
}

// The whole 128-lane image by one warp: four passes of 32 lanes, all loads before all stores
// (the compiler cannot tell the two shared-memory regions apart and would serialise them).
__device__ __forceinline__ void build_metadata_image(const uint8_t* raw_rows, uint8_t* hw_tile, int lane, int rows_used) {
  const uint32_t sel = (lane & 8) ? 0x7632u : 0x5410u;
  const uint4 k01 = make_uint4(0x44444444u, 0x44444444u, 0x44444444u, 0x44444444u);
  uint4 lo[4], hi[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int tl = 32 * i + lane;
    const int row_a = ((tl >> 4) << 4) + (tl & 7), row_b = row_a + 8;
    lo[i] = k01;
    hi[i] = k01;
    if (row_a < rows_used) lo[i] = *(const uint4*)(raw_rows + row_a * 16);
    if (row_b < rows_used) hi[i] = *(const uint4*)(raw_rows + row_b * 16);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint4 a = lo[i], b = hi[i];
    *(uint4*)(hw_tile + (32 * i + lane) * 16) =
        make_uint4(well_formed(prmt(a.x, b.x, sel)), well_formed(prmt(a.y, b.y, sel)),
                   well_formed(prmt(a.z, b.z, sel)), well_formed(prmt(a.w, b.w, sel)));
  }
}

// Fused pruning of one eighth of a pixel row of a stage (the unit of work the pruning threads share
// out): the row's 128 dense channels lie in two 128-byte-swizzled boxes of 64; 16 of them = two
// vectors become one 16-byte chunk of the compressed row, written straight into the A tile's swizzled
// row, and two of the row's sixteen bytes of position metadata (row-major form, as the rearrangement
// step expects). vbase = number of the row's first 8-element vector in the whole dL/dO tensor (random keys).
template <int M, int N, int SCHEME>
__device__ __forceinline__ void fused_prune_eighth(const uint8_t* raw, int a_bytes, uint8_t* a_tile, uint8_t* meta_rows,
                                                   int i, int e, int64_t vbase, uint32_t seed_lo, uint32_t seed_hi) {
  const int sw = i & 7;
  uint4 w[2], out;
#pragma unroll
  for (int jj = 0; jj < 2; ++jj) {
    const int j = 2 * e + jj;
    w[jj] = *(const uint4*)(raw + (j >> 3) * a_bytes + i * 128 + (((j & 7) ^ sw) << 4));
  }
  uint32_t pos[2];
  KeepFlags ka, kb;
  compress_pair<M, N, SCHEME, false>(w[0], w[1], vbase + 2 * e, seed_lo, seed_hi, 0, 0u, out, pos[0], pos[1], ka, kb);
  *(uint4*)(a_tile + i * 128 + ((e ^ sw) << 4)) = out;
  *(uint16_t*)(meta_rows + i * 16 + 2 * e) = (uint16_t)prmt(pos[0], pos[1], 0x0073);
}

template <bool SPARSE, int BN, bool FUSED>
__global__ void __launch_bounds__(FUSED ? kThreadsGemmFused : kThreadsGemm, 1)
dgrad_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmE,
             const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmD,
             const DgradParams p) {
  using C = Cfg<SPARSE, BN>;
  extern __shared__ uint8_t smem_raw[];
  // 1024-byte alignment: required by the 128-byte swizzle of the A, B and staging tiles
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sA = smem;
  uint8_t* sB = smem + p.off_b;
  uint8_t* sEraw = smem + p.off_eraw;
  uint8_t* sEhw = smem + p.off_ehw;
  uint8_t* sW = smem + p.off_w;
  uint8_t* sOut = smem + p.off_out;
  uint8_t* sRaw = smem + p.off_raw;
  uint64_t* full = (uint64_t*)(smem + p.off_bar);
  uint64_t* empty = full + kMaxStages;
  uint64_t* meta_full = empty + kMaxStages;
  uint64_t* acc_full = meta_full + kMaxStages;
  uint64_t* acc_empty = acc_full + 2;
  uint64_t* w_full = acc_empty + 2;
  uint64_t* meta_free = w_full + 1;
  uint64_t* raw_full = meta_free + 2;
  uint32_t* tmem_slot = (uint32_t*)(raw_full + kMaxStages);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = ptx::cluster_ctarank();  // 0: issues the MMAs
  unsigned int* err = &g_device_error;
  const int STAGES = p.stages;
  const int NACC = p.nacc;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxStages; ++s) {
      // full: the producer's arrival (with the stage's byte count) plus, for sparse A, the
      // arrivals of the warps that built the stage's metadata images in both CTAs (one warp per
      // CTA; all four when they also prune) - the MMA thread waits once per stage
      ptx::mbar_init(&full[s], SPARSE ? (FUSED ? 9 : 3) : 1);
      ptx::mbar_init(&empty[s], 1);
      ptx::mbar_init(&meta_full[s], 1);
      ptx::mbar_init(&raw_full[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      ptx::mbar_init(&acc_full[a], 1);
      ptx::mbar_init(&acc_empty[a], 8);
      ptx::mbar_init(&meta_free[a], 8);
    }
    ptx::mbar_init(w_full, 1);
    ptx::fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    ptx::prefetch_tensormap(&tmA);
    ptx::prefetch_tensormap(&tmB);
    if (SPARSE) ptx::prefetch_tensormap(&tmE);
  }
  if (warp == 1) {
    ptx::tmem_alloc_pair(tmem_slot, kTmemCols);
    ptx::tmem_relinquish_pair();
  }
  ptx::tc_fence_before_sync();
  ptx::cluster_sync();  // barrier inits and TMEM of both CTAs are ready before any cross-CTA signal
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  // everything above touched no global memory; the previous kernel's results are needed from here on
  ptx::wait_for_previous_grid();
  // Only now may the next kernel of the stream be scheduled: every CTA of this grid owns its TMEM
  // and has passed its cluster barrier and its wait for the previous grid, so a younger grid can
  // never sit between this grid and a resource it still needs, and at most one grid is resident
  // behind a running one. The younger grid's own TMEM allocation then simply waits for this grid
  // to free its columns, which it does without anyone's help.
  if (p.early) ptx::launch_dependents();

  const int rows_used = p.TW * p.TH * p.TB;
  const int taps = p.R * p.S;
  const bool reuse = (p.rr == p.R) && p.R > 1;
  auto filter_tap = [&p](int r, int s) { return (p.r_first + p.r_step * r) * p.S_full + p.s_first + p.s_step * s; };
  const int groups = reuse ? p.S : taps;  // stage uses per channel block and tile
  const int uses_per_tile = groups * p.k_blocks;
  const int pair_stride = gridDim.x >> 1;
  const int first_pair = blockIdx.x >> 1;
  const int my_tiles = first_pair < p.pair_tiles ? (p.pair_tiles - first_pair + pair_stride - 1) / pair_stride : 0;
  const int n_half = (int)rank * C::kBCols;  // this CTA's column offset inside the BN block

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (ptx::elect_one()) {
      bool alive = true;
      if (p.w_resident) {
        // the layer's whole W half-slice, once: [tap][channel block][box] tiles of kKB rows
        if (rank == 0) ptx::mbar_arrive_expect_tx(w_full, 2u * (uint32_t)(taps * p.k_blocks * C::kTapBBytes));
        for (int t = 0; t < taps; ++t) {
          const int ft = filter_tap(t / p.S, t % p.S);
          for (int cb = 0; cb < p.k_blocks; ++cb)
#pragma unroll
            for (int j = 0; j < C::kBoxes; ++j)
              ptx::tma_load_2d_pair(sW + ((t * p.k_blocks + cb) * C::kBoxes + j) * C::kBoxBytes, &tmB, w_full,
                                    ft * p.Cin + n_half + C::kBoxCols * j, cb * C::kKB);
        }
      }
      const uint32_t pair_tx =
          2u * (uint32_t)((FUSED ? 0 : p.img_rows * 128) + (p.w_resident ? 0 : p.rr * C::kTapBBytes));
      const uint32_t meta_tx = (uint32_t)(p.img_rows * 16);
      int st = 0;
      uint32_t ph = 0;
      for (int pt = first_pair; alive && pt < p.pair_tiles; pt += pair_stride) {
        const int nt = pt % p.tiles_n;
        int t = 2 * (pt / p.tiles_n) + (int)rank;  // this CTA's patch; may lie past the last one
        const int wt = t % p.tiles_w; t /= p.tiles_w;
        const int ht = t % p.tiles_h; t /= p.tiles_h;
        const int bt = t;
        const int n0 = nt * BN + n_half;
        const int cb0 = first_k_block(p, nt * BN, C::kKB);
        const int w0 = wt * p.TW, h0 = ht * p.TH, b0 = bt * p.TB;
        // reuse: a group is the horizontal tap s and the image starts R-1 rows above the row
        // the last vertical tap needs; otherwise a group is the single tap (r, s).
        int r = reuse ? (p.R - 1) : 0, s = 0;
        for (int g = 0; alive && g < groups; ++g) {
          const int q0 = w0 + p.pad_w - s, p0 = h0 + p.pad_h - r;
          for (int cb = 0; cb < p.k_blocks; ++cb) {
            if (!ptx::mbar_wait(&empty[st], ph ^ 1u, err, 0x100u + st)) { alive = false; break; }
            if (rank == 0) ptx::mbar_arrive_expect_tx(&full[st], pair_tx);
            if (FUSED) {
              // dense dL/dO of this CTA's patch: 128 channels as two boxes of 64
              ptx::mbar_arrive_expect_tx(&raw_full[st], 2u * (uint32_t)(p.img_rows * 128));
              ptx::tma_load_4d(sRaw + st * 2 * p.a_bytes, &tmA, &raw_full[st], (cb0 + cb) * 128, q0, p0, b0);
              ptx::tma_load_4d(sRaw + st * 2 * p.a_bytes + p.a_bytes, &tmA, &raw_full[st], (cb0 + cb) * 128 + 64, q0, p0, b0);
            } else {
              if (SPARSE) {
                ptx::mbar_arrive_expect_tx(&meta_full[st], meta_tx);
                ptx::tma_load_4d(sEraw + st * p.eraw_bytes, &tmE, &meta_full[st], (cb0 + cb) * 8, q0, p0, b0);
              }
              ptx::tma_load_4d_pair(sA + st * p.a_bytes, &tmA, &full[st], (cb0 + cb) * 64, q0, p0, b0);
            }
            if (!p.w_resident) {
              for (int u = 0; u < p.rr; ++u) {
                const int tap = filter_tap(reuse ? u : r, s);
#pragma unroll
                for (int j = 0; j < C::kBoxes; ++j)
                  ptx::tma_load_2d_pair(sB + st * p.b_bytes + (u * C::kBoxes + j) * C::kBoxBytes, &tmB, &full[st],
                                        tap * p.Cin + n0 + C::kBoxCols * j, (cb0 + cb) * C::kKB);
              }
            }
            if (++st == STAGES) { st = 0; ph ^= 1u; }
          }
          if (++s == p.S) { s = 0; if (!reuse) ++r; }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------- MMA issuer (first CTA only)
    // A single thread executes roughly one dependent instruction per ten clocks, so its path
    // per stage is short: one barrier wait, descriptor words kept as running sums.
    if (rank == 0 && ptx::elect_one()) {
      const uint32_t idesc = make_idesc(BN, SPARSE) & ~(p.f16 ? kIdescBf16Operands : 0u);
      bool alive = true;
      if (p.w_resident) alive = ptx::mbar_wait(w_full, 0u, err, 0x700u);
      // descriptors as two 32-bit halves: the start address only ever changes the low word
      const uint64_t adesc0 = ptx::make_smem_desc(0, 16, 1024, 2);
      const uint64_t bdesc0 = ptx::make_smem_desc(0, C::kBoxBytes, 8 * C::kRowB, C::kBSwizzle);
      const uint64_t edesc0 = ptx::make_smem_desc(0, 128, 128, 0);
      const uint32_t a_hi = (uint32_t)(adesc0 >> 32), b_hi = (uint32_t)(bdesc0 >> 32), e_hi = (uint32_t)(edesc0 >> 32);
      const uint32_t a_lo0 = (uint32_t)adesc0 + (ptx::smem_u32(sA) >> 4);
      const uint32_t b_lo0 = (uint32_t)bdesc0 + (ptx::smem_u32(sB) >> 4);
      const uint32_t w_lo0 = (uint32_t)bdesc0 + (ptx::smem_u32(sW) >> 4);
      const uint32_t e_lo0 = (uint32_t)edesc0 + (ptx::smem_u32(sEhw) >> 4);
      const uint32_t a_stage16 = (uint32_t)p.a_bytes >> 4, b_stage16 = (uint32_t)p.b_bytes >> 4,
                     e_stage16 = (uint32_t)p.ehw_bytes >> 4;
      constexpr uint32_t kTapB16 = (uint32_t)C::kTapBBytes >> 4;
      constexpr uint32_t kBStep = (uint32_t)((C::kKB / 4) * C::kRowB / 16);  // W rows of one MMA
      const uint32_t slot_cols = 4u * (uint32_t)p.rr;                         // metadata columns of one stage
      int st = 0, acc = 0;
      uint32_t ph = 0, aph = 0;
      uint32_t a_lo = a_lo0, b_lo = b_lo0, e_lo = e_lo0, mcol = 0;  // running words of the stage ring
      for (int lt = 0; alive && lt < my_tiles; ++lt) {
        if (!ptx::mbar_wait(&acc_empty[acc], aph ^ 1u, err, 0x200u + acc)) break;
        // Shared metadata region: this tile's slots are the first columns of the other
        // accumulator, which the epilogue of the previous tile must have read out first.
        if (p.meta_shared && lt > 0 &&
            !ptx::mbar_wait(&meta_free[acc ^ 1], (((uint32_t)lt - 1u) >> 1) & 1u, err, 0x800u + acc))
          break;
        const uint32_t meta_base = tmem_base + (uint32_t)(p.meta_shared ? (acc ^ 1) * BN : p.meta_col);
        ptx::tc_fence_after_sync();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
        uint32_t accumulate = 0u;
        // This thread's instructions set the pace of narrow tiles (65 x 2688 . 2688 x 576: 20 ns more per block with a test for partial
        // blocks in it). WHOLE: every channel block is, and the loop holds no such test; else the layer's last block may be partial.
        auto tile = [&](auto whole_tag) {
          constexpr bool WHOLE = decltype(whole_tag)::value;
          int cb_last = 0;  // the partial block's place in the tile's window
          if (!WHOLE) {
            cb_last = p.k_last;
            if (p.diag_cin_g != 0) cb_last -= first_k_block(p, (first_pair + lt * pair_stride) % p.tiles_n * BN, C::kKB);
          }
          int r_single = 0, s = 0;
          for (int g = 0; alive && g < groups; ++g) {
            for (int cb = 0; cb < p.k_blocks; ++cb) {
              if (!ptx::mbar_wait(&full[st], ph, err, 0x300u + st)) { alive = false; break; }
              ptx::tc_fence_after_sync();
              const uint32_t e_col = meta_base + mcol;  // even: slots are multiples of 4 columns apart
              const int mmas = !WHOLE && cb == cb_last ? p.last_mmas : 4;
              if (SPARSE) {
                for (int u = 0; u < p.rr; ++u)
                  ptx::tc_cp_128x128b_pair(e_col + 4u * u, ((uint64_t)e_hi << 32) | (e_lo + (uint32_t)(u * (kEHwBytes / 16))));
              }
              for (int u = 0; u < p.rr; ++u) {
                // vertical tap r: the tile's rows start (R-1-r) image rows into the stage
                const int r = reuse ? u : r_single;
                const uint32_t a_u = a_lo + (reuse ? (uint32_t)((p.R - 1 - r) * p.TW * 8) : 0u);
                const uint32_t b_u = p.w_resident ? w_lo0 + (uint32_t)((r * p.S + s) * p.k_blocks + cb) * kTapB16
                                                  : b_lo + (uint32_t)u * kTapB16;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                  if (!WHOLE && q >= mmas) break;
                  // A: 32 bytes of a 128-byte swizzled row per MMA; B: 16 (dense) or 32 (sparse) rows
                  const uint64_t a_q = ((uint64_t)a_hi << 32) | (a_u + (uint32_t)(q * 2));
                  const uint64_t b_q = ((uint64_t)b_hi << 32) | (b_u + (uint32_t)q * kBStep);
                  if (SPARSE)
                    ptx::mma_sp_f16_ss_pair(d_tmem, a_q, b_q, e_col + 4u * u + (uint32_t)(q & 2), idesc | (uint32_t)(q & 1),
                                            q == 0 ? accumulate : 1u);
                  else
                    ptx::mma_f16_ss_pair(d_tmem, a_q, b_q, idesc, q == 0 ? accumulate : 1u);
                }
                accumulate = 1u;
              }
              ptx::tc_commit_pair(&empty[st], 3);
              if (++st == STAGES) { st = 0; ph ^= 1u; a_lo = a_lo0; b_lo = b_lo0; e_lo = e_lo0; mcol = 0; }
              else { a_lo += a_stage16; b_lo += b_stage16; e_lo += e_stage16; mcol += slot_cols; }
            }
            if (++s == p.S) { s = 0; ++r_single; }
          }
        };
        if (p.last_mmas == 4) tile(std::true_type{});
        else tile(std::false_type{});
        if (alive) ptx::tc_commit_pair(&acc_full[acc], 3);
        if (++acc == NACC) { acc = 0; aph ^= 1u; }
      }
    }
  } else if (warp < 6 || warp >= 10) {  // warps 10.. exist only in the fused instantiation
    // ------------------------------------------------- metadata rearranger
    if (SPARSE && !FUSED) {
      // A lone warp runs a dependent chain slowly, so the four warps do not share a stage: warp k
      // owns stages k, k+G, ... of the ring and builds the TMEM metadata images of every use of
      // those stages (four passes of 32 lanes per image); consecutive uses fall to different warps,
      // so up to G are in flight.
      // Ownership goes by STAGE, not by use: a parity wait tells "the phase I expect has completed"
      // from "the phase two before it has" only if the waiter saw the phase in between complete.
      // The warp that owns a stage waits for each of its uses in turn, so it always has. (A warp
      // that took uses k, k+G, ... regardless of stage would wait for use u of a stage without
      // having waited for use u - STAGES; that box was requested earlier than the boxes the warp
      // did see land, but TMA boxes may land out of request order, and a box that is late lets
      // the wait pass one phase early.)
      const int G = STAGES < 4 ? STAGES : 4;
      const int total_uses = (warp - 2 < G) ? my_tiles * uses_per_tile : 0;
      uint32_t ph = 0;
      for (int first = 0; first < total_uses; first += STAGES, ph ^= 1u) {  // one pass over the ring
        bool alive = true;
        for (int st = warp - 2; st < STAGES && first + st < total_uses; st += G) {
          // the metadata box was requested after the stage's previous use had been consumed
          if (!ptx::mbar_wait(&meta_full[st], ph, err, 0x500u + st)) { alive = false; break; }
          for (int v = 0; v < p.rr; ++v) {
            const int row_off = reuse ? (p.R - 1 - v) * p.TW : 0;
            build_metadata_image(sEraw + st * p.eraw_bytes + row_off * 16, sEhw + st * p.ehw_bytes + v * kEHwBytes, lane,
                                 rows_used);
          }
          ptx::fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive_cluster(&full[st], 0);
        }
        if (!alive) break;
      }
    } else if (SPARSE) {
      // Fused pruning: warps 2..5 and the helper warps 10.. share out the stage's pixel rows in eighths
      // (item = row, eighth); then each thread of warps 2..5 builds one TMEM lane of every metadata image.
      const int pruner = warp < 6 ? (int)threadIdx.x - 64 : 128 + (int)threadIdx.x - kThreadsGemm;  // 0 .. kFusedPruners - 1
      const int row = threadIdx.x - 64;  // warps 2..5 only
      bool alive = true;
      int st = 0;
      uint32_t ph = 0;
      const int img_h = p.TH + p.rr - 1;
      for (int pt = first_pair; alive && pt < p.pair_tiles; pt += pair_stride) {
        int t = 2 * (pt / p.tiles_n) + (int)rank;
        const int wt = t % p.tiles_w; t /= p.tiles_w;
        const int ht = t % p.tiles_h; t /= p.tiles_h;
        const int w0 = wt * p.TW, h0 = ht * p.TH, b0 = t * p.TB;
        const int cb0 = first_k_block(p, (pt % p.tiles_n) * BN, C::kKB);
        int r = reuse ? (p.R - 1) : 0, s = 0, cb = 0;
        for (int k = 0; k < uses_per_tile; ++k) {
          // the pruning warps stay or leave together: they meet at a named barrier below
          if (!ptx::named_bar_all(2, kFusedPruners, ptx::mbar_wait(&raw_full[st], ph, err, 0x900u + st))) { alive = false; break; }
          const int q0 = w0 + p.pad_w - s, p0 = h0 + p.pad_h - r;
          const uint8_t* raw = sRaw + st * 2 * p.a_bytes;
          uint8_t* a_tile = sA + st * p.a_bytes;
          uint8_t* meta_rows = sEraw + st * p.eraw_bytes;
          for (int item = pruner; item < 8 * p.img_rows; item += kFusedPruners) {
            const int i = item >> 3, e = item & 7;
            const int iw = i % p.TW, ih = (i / p.TW) % img_h, ib = i / (p.TW * img_h);
            const int64_t pixel = ((int64_t)(b0 + ib) * p.P + (p0 + ih)) * p.Q + (q0 + iw);  // any value when outside
            const int64_t vbase = pixel * (p.Cout >> 3) + (cb0 + cb) * 16;
#define SDGP_FUSED_ITEM(MM, NN, SS) fused_prune_eighth<MM, NN, SS>(raw, p.a_bytes, a_tile, meta_rows, i, e, vbase, p.seed_lo, p.seed_hi)
#define SDGP_FUSED_M(MM)                                                                                                   \
  if (p.fused_scheme == SDGP_MAGNITUDE) { if (p.fused_n == 1) SDGP_FUSED_ITEM(MM, 1, SDGP_MAGNITUDE); else SDGP_FUSED_ITEM(MM, 2, SDGP_MAGNITUDE); } \
  else if (p.fused_scheme == SDGP_RANDOM) { if (p.fused_n == 1) SDGP_FUSED_ITEM(MM, 1, SDGP_RANDOM); else SDGP_FUSED_ITEM(MM, 2, SDGP_RANDOM); }    \
  else { if (p.fused_n == 1) SDGP_FUSED_ITEM(MM, 1, SDGP_RESCALED_MAGNITUDE); else SDGP_FUSED_ITEM(MM, 2, SDGP_RESCALED_MAGNITUDE); }
            if (p.fused_m == 4) { SDGP_FUSED_M(4) } else if (p.fused_m == 8) { SDGP_FUSED_M(8) } else { SDGP_FUSED_M(16) }
#undef SDGP_FUSED_M
#undef SDGP_FUSED_ITEM
          }
          ptx::fence_proxy_async_smem();                // the compressed tile is read by the tensor core
          ptx::named_bar_sync(2, kFusedPruners);        // every row's metadata is in place before it is rearranged
          if (warp < 6) {
            for (int u = 0; u < p.rr; ++u) {
              const int row_off = reuse ? (p.R - 1 - u) * p.TW : 0;
              build_metadata_lane(sEraw + st * p.eraw_bytes + row_off * 16, sEhw + st * p.ehw_bytes + u * kEHwBytes, row,
                                  rows_used);
            }
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_cluster(&full[st], 0);
          }
          if (++st == STAGES) { st = 0; ph ^= 1u; }
          if (++cb == p.k_blocks) {
            cb = 0;
            if (++s == p.S) { s = 0; if (!reuse) ++r; }
          }
        }
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue
    const int q = warp & 3;  // a warp may only touch TMEM lanes [32*(warp%4), +32)
    const int row = q * 32 + lane;
    const int iw = row % p.TW, ih = (row / p.TW) % p.TH, ib = row / (p.TW * p.TH);  // this thread's pixel of a patch
    uint32_t aph = 0, chunk = 0;
    int acc = 0;
    for (int pt = first_pair; pt < p.pair_tiles; pt += pair_stride) {
      const int n0 = (pt % p.tiles_n) * BN;
      const int mt = 2 * (pt / p.tiles_n) + (int)rank;
      int t = mt;
      const int w = (t % p.tiles_w) * p.TW + iw; t /= p.tiles_w;
      const int h = (t % p.tiles_h) * p.TH + ih; t /= p.tiles_h;
      const int b = t * p.TB + ib;
      if (!ptx::mbar_wait(&acc_full[acc], aph, err, 0x600u + acc)) break;
      ptx::tc_fence_after_sync();
      const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN);
      uint64_t* first_slab_read = p.meta_shared ? &meta_free[acc] : nullptr;
      if (p.box_store) {
        store_box<BN>(taddr, sOut + q * p.out_bufs * kSlabBytes, &tmD, false, n0, w - lane, h, b, 0, mt < p.m_tiles, p.d.channels - n0,
                      first_slab_read, &acc_empty[acc], p.f16 != 0, p.out_bufs, chunk);
      } else {
        const bool inside = row < rows_used && mt < p.m_tiles && w < p.W && h < p.H && b < p.B;
        uint8_t* dst = inside ? p.d.base + b * p.d.sb + h * p.d.sh + w * p.d.sw + 2 * n0 : nullptr;
        store_rows<BN>(taddr, dst, p.d.channels - n0, p.d.aligned32 != 0, first_slab_read, &acc_empty[acc], p.f16 != 0);
      }
      if (++acc == NACC) { acc = 0; aph ^= 1u; }
    }
    // the staging rows have been read; the writes themselves complete with the grid (whoever depends on dD waits for that)
    if (lane == 0) ptx::bulk_wait_group_read<0>();
  }

  __syncwarp();
  if (*(volatile unsigned int*)err != 0u) {
    // A wait gave up somewhere: loads may still be in flight towards this CTA's shared
    // memory. Give them a bounded while to land before the CTA goes away.
    const uint64_t t0 = ptx::globaltimer_ns();
    while (ptx::globaltimer_ns() - t0 < 200000ull) {
    }
  }
  ptx::tc_fence_before_sync();
  __syncwarp();
  ptx::cluster_sync();  // neither CTA leaves (or frees TMEM) while the other may still touch it
  ptx::tc_fence_after_sync();
  if (warp == 1) ptx::tmem_dealloc_pair(tmem_base, kTmemCols);
}

// Shared-memory plan for one launch: decides filter-row reuse, resident W, pipeline depth,
// accumulator count and the carve. Returns false if no variant fits.
template <bool SPARSE, int BN, bool FUSED>
bool plan(DgradParams* p) {
  using C = Cfg<SPARSE, BN>;
  const int taps = p->R * p->S;
  const int budget = kSmemLimit - kSmemSlack;
  // Boxes where a warp's 32 rows are 32 pixels of one image row and the epilogues overlap other tiles (store_box); rows where
  // the only epilogue of a CTA pair is the tail of the launch.
  p->box_store = (p->TW == kBM && p->pair_tiles > kBoxStoreRounds * (sm_count() / 2)) ? 1 : 0;
  // Filter-row reuse needs a single-image patch whose rows are whole groups of 8 pixels, so
  // that every vertical tap is an offset of whole 1024-byte swizzle periods.
  const bool can_reuse = p->R > 1 && p->TB == 1 && p->TW % 8 == 0 && p->TW * (p->TH + p->R - 1) <= kMaxImgRows;
  const bool can_reside = p->tiles_n == 1 && p->diag_cin_g == 0 && p->pair_tiles > sm_count() / 2;  // pays only if tiles repeat
  for (int attempt = 0; attempt < 4; ++attempt) {
    // attempt 0: reuse with streamed W (measured best where it fits: more stages in flight),
    // 1: reuse + resident W, 2: resident W, 3: neither
    const bool reuse = attempt < 2;
    const bool resident = (attempt == 1 || attempt == 2);
    if ((reuse && !can_reuse) || (resident && !can_reside)) continue;
    p->rr = reuse ? p->R : 1;
    p->img_rows = p->TW * (p->TH + p->rr - 1) * p->TB;
    p->w_resident = resident ? 1 : 0;
    p->a_bytes = round_up(p->img_rows * 128, 1024);
    p->b_bytes = resident ? 0 : p->rr * C::kTapBBytes;
    p->eraw_bytes = SPARSE ? round_up(p->img_rows * 16, 128) : 0;
    p->ehw_bytes = SPARSE ? p->rr * kEHwBytes : 0;
    const int w_bytes = resident ? taps * p->k_blocks * C::kTapBBytes : 0;
    const int raw_bytes = FUSED ? 2 * p->a_bytes : 0;
    const int stage_bytes = p->a_bytes + p->b_bytes + p->eraw_bytes + p->ehw_bytes + raw_bytes;
    p->out_bufs = p->box_store ? 2 : 0;
    int out_bytes = 4 * p->out_bufs * kSlabBytes;
    int stages = (budget - w_bytes - out_bytes) / stage_bytes;
    if (p->box_store && stages < 4) {
      p->out_bufs = 1;
      out_bytes = 4 * kSlabBytes;
      stages = (budget - w_bytes - out_bytes) / stage_bytes;
    }
    if (stages > kMaxStages) stages = kMaxStages;
    // TMEM: accumulators first, metadata slots (4 columns per tap and stage) behind them
    const int meta_cols_per_stage = SPARSE ? 4 * p->rr : 0;
    const int meta_div = SPARSE ? meta_cols_per_stage : 1;  // divisor that is never zero
    int nacc = (2 * BN + 2 * meta_cols_per_stage <= (int)kTmemCols) ? 2 : 1;
    p->meta_shared = 0;
    if (meta_cols_per_stage > 0 && nacc == 1 && 2 * BN <= (int)kTmemCols) {
      // Two accumulators fill TMEM: the metadata slots share the first 64 columns of whichever
      // accumulator is being read out, released early by the epilogue.
      nacc = 2;
      p->meta_shared = 1;
      if (stages > 64 / meta_div) stages = 64 / meta_div;
    } else if (meta_cols_per_stage > 0) {
      const int max_meta_stages = ((int)kTmemCols - nacc * BN) / meta_div;
      if (stages > max_meta_stages) stages = max_meta_stages;
    }
    p->nacc = nacc;
    p->meta_col = p->meta_shared ? 0 : nacc * BN;
    for (; stages >= ((resident || reuse || FUSED) ? 2 : 3); --stages) {  // (a reuse stage is R taps long)
      p->stages = stages;
      p->off_b = stages * p->a_bytes;
      p->off_eraw = p->off_b + stages * p->b_bytes;
      p->off_ehw = round_up(p->off_eraw + stages * p->eraw_bytes, 1024);
      p->off_w = round_up(p->off_ehw + stages * p->ehw_bytes, 1024);
      p->off_out = round_up(p->off_w + w_bytes, 1024);
      p->off_raw = p->off_out + out_bytes;
      p->off_bar = p->off_raw + stages * raw_bytes;
      p->smem_bytes = p->off_bar + 512 + 1024;
      if (p->smem_bytes <= kSmemLimit) return true;  // (the sections' alignment may cost a stage)
    }
  }
  return false;
}

template <bool SPARSE, int BN, bool FUSED>
sdgp_status launch_cfg(const void* A, const void* meta, const void* Wt, const DgradView& view, DgradParams p,
                       cudaStream_t stream) {
  const int P = view.P, Q = view.Q;
  using C = Cfg<SPARSE, BN>;
  if (!plan<SPARSE, BN, FUSED>(&p)) return SDGP_ERR_UNSUPPORTED;
  p.d = view.d;
  p.early = early_for(SPARSE && !FUSED && p.last_launch, pairs_for(p.pair_tiles));

  CUtensorMap tmA, tmE, tmB, tmD;
  const uint32_t img_h = (uint32_t)(p.TH + p.rr - 1);
  const uint64_t CA = (SPARSE && !FUSED) ? (uint64_t)view.a_channels / 2 : (uint64_t)view.a_channels;  // stored elements per pixel
  {
    const uint64_t dims[4] = {CA, (uint64_t)Q, (uint64_t)P, (uint64_t)view.batch};
    const uint64_t strides[3] = {CA * 2, CA * 2 * Q, CA * 2 * Q * P};
    const uint32_t box[4] = {64, (uint32_t)p.TW, img_h, (uint32_t)p.TB};
    if (!encode(&tmA, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, A, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B))
      return SDGP_ERR_CUDA;
  }
  if (SPARSE && !FUSED) {
    const uint64_t CE = (uint64_t)view.meta_channels / 16;
    const uint64_t dims[4] = {CE, (uint64_t)Q, (uint64_t)P, (uint64_t)view.batch};
    const uint64_t strides[3] = {CE * 2, CE * 2 * Q, CE * 2 * Q * P};
    const uint32_t box[4] = {8, (uint32_t)p.TW, img_h, (uint32_t)p.TB};
    if (!encode(&tmE, CU_TENSOR_MAP_DATA_TYPE_UINT16, 4, meta, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_NONE))
      return SDGP_ERR_CUDA;
  } else {
    tmE = tmA;
  }
  {
    const uint64_t dims[2] = {(uint64_t)view.w_cols, (uint64_t)p.Cout};
    const uint64_t strides[1] = {(uint64_t)view.w_cols * 2};
    const uint32_t box[2] = {(uint32_t)C::kBoxCols, (uint32_t)C::kKB};
    if (!encode(&tmB, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Wt, dims, strides, box,
                C::kRowB == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B))
      return SDGP_ERR_CUDA;
  }
  tmD = tmA;
  if (p.box_store) {
    const uint64_t dims[4] = {(uint64_t)p.d.channels, (uint64_t)p.W, (uint64_t)p.H, (uint64_t)p.B};
    const uint64_t strides[3] = {(uint64_t)p.d.sw, (uint64_t)p.d.sh, (uint64_t)p.d.sb};
    const uint32_t box[4] = {64, 32, 1, 1};
    if (!encode(&tmD, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, p.d.base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B))
      return SDGP_ERR_CUDA;
  }
  static bool configured[kMaxDevices] = {};
  auto kernel = dgrad_kernel<SPARSE, BN, FUSED>;
  if (!configure_once(kernel, configured)) return SDGP_ERR_CUDA;
  return launch_pairs(kernel, pairs_for(p.pair_tiles), FUSED ? kThreadsGemmFused : kThreadsGemm, p.smem_bytes, stream, tmA, tmE, tmB, tmD, p);
}

template <bool SPARSE, bool FUSED>
sdgp_status launch_bn(int bn, const void* A, const void* meta, const void* Wt, const DgradView& view, const DgradParams& p,
                      cudaStream_t stream) {
  switch (bn) {
    case 64: return launch_cfg<SPARSE, 64, FUSED>(A, meta, Wt, view, p, stream);
    case 128: return launch_cfg<SPARSE, 128, FUSED>(A, meta, Wt, view, p, stream);
    case 192: return launch_cfg<SPARSE, 192, FUSED>(A, meta, Wt, view, p, stream);
    default: return launch_cfg<SPARSE, 256, FUSED>(A, meta, Wt, view, p, stream);
  }
}

}  // namespace

sdgp_status launch_general(bool sparse, bool fused, int bn, const void* A, const void* meta, const void* Wt, const DgradView& view,
                           const DgradParams& p, cudaStream_t stream) {
  if (fused) return launch_bn<true, true>(bn, A, meta, Wt, view, p, stream);
  return sparse ? launch_bn<true, false>(bn, A, meta, Wt, view, p, stream) : launch_bn<false, false>(bn, A, meta, Wt, view, p, stream);
}

cudaError_t take_error_general(unsigned int* word) { return take_error_word(word); }

}  // namespace sdgp
