// Fused prune + contraction for grouped convolutions with narrow groups (the 3 x 3 convolutions of RegNetX, Section 4): 16 or 32
// channels per group on both sides.
//
// Such a layer is memory-bound: a group's products are few (16 x 16 per tap and pixel), so dL/dO is read once, pruned on its way into
// shared memory, multiplied there and never stored. The other path (prune kernel, block-diagonal filters, contraction of
// 128-channel blocks) multiplies 8 times as many zeros and makes three launches of it.
//
// Raster. The pixels of all images are laid out in one line: rows of `pitch` positions, `img_pos` positions an image, with as many zero
// positions behind each row and each image as a filter tap can reach past it (the zeros behind one row are also the ones before the next).
// A tap is then ONE offset in that line for every pixel, whatever the image size: the operand of a tap is 128 consecutive rows of
// shared memory, starting at any row (the matrix descriptor swizzles by absolute address bits). 14 x 14 images fill 87 % of the
// accumulator rows this way, strips of 8 x 16 pixels 77 %. Stride 2 is four stride-1 problems, one per output parity, over the
// same line: the four classes share the pruned operand and have an accumulator each.
//
// Work unit: 64 channels (64 / group width groups) of up to 128 * tiles consecutive positions. Warp roles (24 warps): warp 0 streams dL/dO
// and warp 2 the filters by TMA, warp 1 issues the MMAs (128 x width x 16, one group at a time), warps 4..7 are the epilogue, the other
// seventeen prune: a thread takes two vectors of 8 channels out of the stage that TMA filled and puts them back pruned, dense, for the
// tensor core. Dense, because the MMA's time is reading its 128 rows of A (4 KB: 41 clocks at best) for either kind and 16 columns leave the
// tensor pipe idle anyway. A pruned position is thus a zero that meets its filter, where the compressed form skips it: with filters that are not
// finite the two differ. (Loading dL/dO into the pruning warps' registers instead measured the same within 3 %.) 256 images of 14 x 14, 10 groups of 16, rescaled, us: three kernels 32.8, this 22.8; 124 x 4 x 4, 11 groups, 11.2 and
// 5.2; 60 x 32 x 32, 15 groups, 31.7 and 26.5. What bounds it: the pruning of the random and rescaled functions - the first layer's units take some 4600
// clocks of it, halo positions (a fifth there, 40 % at 32 x 32) and the absent half of the last block of 32 channels included - beside MMAs of
// 51 to 59 clocks each, 4000 a unit, half of that in the last block. 80 registers are the most 24 warps can have; the pruning spills 32 to 40 bytes.
#include "dgrad_prune.cuh"

namespace sdgp {
namespace {

constexpr int kGrThreads = 24 * 32;
constexpr int kGrPruneWarps = 17;
constexpr int kGrMaxStages = 4;  // operand stages
constexpr int kGrMaxTaps = 32;
constexpr int kGrBlock = 64;     // channels of a unit: one 128-byte swizzled row

struct GroupedParams {
  uint8_t* dD;
  int B, P, Q, H, W, C;          // C channels on both sides
  int gw;                        // channels of a group: 16 or 32
  int stride, classes;           // output parities with an accumulator (1, or 4 for stride 2)
  int pitch, img_pos;            // raster
  uint32_t mg_pitch, mg_img;     // div_magic of the two
  int len;                       // positions of all images
  int k_blocks, tiles, units;
  int span;                      // positions of a unit
  uint32_t mg_kb;
  int off_min, reach;            // smallest tap offset; the largest's distance from it
  int chunk_rows, chunk_pos;     // rows of an image (a divisor of its rows in the line) that one TMA box brings; their positions
  uint32_t mg_chunk;
  int taps, class_end[4];        // taps in class order; first tap past each class
  short tap_off[kGrMaxTaps];     // offset of a tap (positions) minus off_min
  short tap_filter[kGrMaxTaps];  // its number in the filter
  int n, m, f16;
  uint32_t seed_lo, seed_hi;
  int aligned32;                 // dD: 32-byte accesses
  int a_stages, a_bytes, w_tap_bytes, w_bytes, off_w, off_bar;
};

// x / d and x % d for a divisor fixed for the launch, m = floor(2^32 / d) (0xFFFFFFFF for d = 1).
__device__ __forceinline__ void gr_divmod(uint32_t x, uint32_t d, uint32_t m, uint32_t& q, uint32_t& r) {
  q = __umulhi(x, m);
  r = x - q * d;
  if (r >= d) { ++q; r -= d; }
}

// Position L >= 0 of the raster -> image, row, column.
__device__ __forceinline__ void gr_locate(const GroupedParams& p, uint32_t L, uint32_t& img, uint32_t& h, uint32_t& w) {
  uint32_t rem;
  gr_divmod(L, (uint32_t)p.img_pos, p.mg_img, img, rem);
  gr_divmod(rem, (uint32_t)p.pitch, p.mg_pitch, h, w);
}

// Keep masks of a vector's four words.
__device__ __forceinline__ uint4 keep_masks(const KeepFlags& k) {
  return make_uint4(prmt(k.k0, k.k1, 0xDD99), prmt(k.k2, k.k3, 0xDD99), prmt(k.k0, k.k1, 0xFFBB), prmt(k.k2, k.k3, 0xFFBB));
}
__device__ __forceinline__ uint4 and4(const uint4& a, const uint4& b) { return make_uint4(a.x & b.x, a.y & b.y, a.z & b.z, a.w & b.w); }
// Sums of the magnitudes of a vector's two halves, in the tree of Algorithm 1's rescale.
template <bool F16>
__device__ __forceinline__ float2 half_sums(const uint4& w) {
  return make_float2(__fadd_rn(pair_abs<F16>(w.x), pair_abs<F16>(w.y)), __fadd_rn(pair_abs<F16>(w.z), pair_abs<F16>(w.w)));
}
__device__ __forceinline__ float rescale_factor(float total, float kept) { return kept == 0.0f ? 1.0f : __fdiv_rn(total, kept); }
template <bool F16>
__device__ __forceinline__ void rescale_vector(uint4& y, const uint4& mask, float lo, float hi, bool finite) {
  y = make_uint4(rescale_slots<F16>(y.x, lo, finite, mask.x), rescale_slots<F16>(y.y, lo, finite, mask.y),
                 rescale_slots<F16>(y.z, hi, finite, mask.z), rescale_slots<F16>(y.w, hi, finite, mask.w));
}

// Two neighbouring vectors (numbers v and v + 1, v even) pruned in place, as Algorithm 1's dense result. A group of 32 channels is held by
// two neighbouring lanes, which call together; part: which half of it this lane has.
template <int M, int N, int SCHEME, bool F16>
__device__ __forceinline__ void prune_dense_pair(uint4& wa, uint4& wb, int64_t v, uint32_t seed_lo, uint32_t seed_hi, int part) {
  KeepFlags ka, kb;
  if constexpr (M == 4) {
    ka = m4_flags<N, SCHEME == SDGP_RANDOM ? SDGP_RANDOM : SDGP_MAGNITUDE>(wa, v, seed_lo, seed_hi);
    kb = m4_flags<N, SCHEME == SDGP_RANDOM ? SDGP_RANDOM : SDGP_MAGNITUDE>(wb, v + 1, seed_lo, seed_hi);
  } else {
    uint32_t ca[8], cb[8], ha, la, hb, lb;
    const uint32_t pos0 = M == 32 ? 31u - 16u * (uint32_t)part : 31u;
    top2_keys<SCHEME>(wa, v, seed_lo, seed_hi, pos0, ca);
    top2_keys<SCHEME>(wb, v + 1, seed_lo, seed_hi, M == 8 ? pos0 : pos0 - 8u, cb);
    top2_of_8(ca, ha, la);
    top2_of_8(cb, hb, lb);
    if (M != 8) {
      merge_top2(ha, la, hb, lb);
      if (M == 32) merge_top2(ha, la, __shfl_xor_sync(0xFFFFFFFFu, ha, 1), __shfl_xor_sync(0xFFFFFFFFu, la, 1));
      hb = ha;
      lb = la;
    }
    ka = top2_flags(ca, (N == 1 ? ha : la) - 1u);
    kb = top2_flags(cb, (N == 1 ? hb : lb) - 1u);
  }
  const uint4 ma = keep_masks(ka), mb = keep_masks(kb), ya = and4(wa, ma), yb = and4(wb, mb);
  if (SCHEME == SDGP_RESCALED_MAGNITUDE) {
    const float2 ta = half_sums<F16>(wa), tb = half_sums<F16>(wb), sa = half_sums<F16>(ya), sb = half_sums<F16>(yb);
    wa = ya;
    wb = yb;
    if (M == 4) {
      rescale_vector<F16>(wa, ma, rescale_factor(ta.x, sa.x), rescale_factor(ta.y, sa.y), is_finite(ta.x) && is_finite(ta.y));
      rescale_vector<F16>(wb, mb, rescale_factor(tb.x, sb.x), rescale_factor(tb.y, sb.y), is_finite(tb.x) && is_finite(tb.y));
    } else {
      float t0 = __fadd_rn(ta.x, ta.y), t1 = __fadd_rn(tb.x, tb.y), s0 = __fadd_rn(sa.x, sa.y), s1 = __fadd_rn(sb.x, sb.y);
      if (M != 8) {
        t0 = __fadd_rn(t0, t1);
        s0 = __fadd_rn(s0, s1);
        if (M == 32) {
          t0 = __fadd_rn(t0, __shfl_xor_sync(0xFFFFFFFFu, t0, 1));
          s0 = __fadd_rn(s0, __shfl_xor_sync(0xFFFFFFFFu, s0, 1));
        }
        t1 = t0;
        s1 = s0;
      }
      const float f0 = rescale_factor(t0, s0), f1 = M == 8 ? rescale_factor(t1, s1) : f0;
      rescale_vector<F16>(wa, ma, f0, f0, is_finite(t0));
      rescale_vector<F16>(wb, mb, f1, f1, is_finite(t1));
    }
  } else {
    wa = ya;
    wb = yb;
  }
}

template <int SCHEME, bool F16>
__global__ void __launch_bounds__(kGrThreads, 1)
grouped_fused_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW, const __grid_constant__ GroupedParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sA = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sW = sA + p.off_w;
  uint64_t* raw_full = (uint64_t*)(sA + p.off_bar);  // TMA has filled the stage
  uint64_t* a_full = raw_full + kGrMaxStages;         // ... and it is pruned
  uint64_t* a_empty = a_full + kGrMaxStages;
  uint64_t* w_full = a_empty + kGrMaxStages;  // two W stages
  uint64_t* w_empty = w_full + 2;
  uint64_t* acc_full = w_empty + 2;
  uint64_t* acc_empty = acc_full + 2;
  uint32_t* tmem_slot = (uint32_t*)(acc_empty + 2);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  unsigned int* err = &g_device_error;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kGrMaxStages; ++s) {
      ptx::mbar_init(&raw_full[s], 1);
      ptx::mbar_init(&a_full[s], kGrPruneWarps);
      ptx::mbar_init(&a_empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      ptx::mbar_init(&w_full[a], 1);
      ptx::mbar_init(&w_empty[a], 1);
      ptx::mbar_init(&acc_full[a], 1);
      ptx::mbar_init(&acc_empty[a], 4);
    }
    ptx::fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    ptx::prefetch_tensormap(&tmA);
    ptx::prefetch_tensormap(&tmW);
  }
  if (warp == 1) {
    ptx::tmem_alloc(tmem_slot, kTmemCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base_any = *tmem_slot;
  ptx::wait_for_previous_grid();
  ptx::launch_dependents();  // (after every wait without a time limit: see the general kernel)

  const int first = blockIdx.x, step = gridDim.x;
  const int acc_cols = p.classes * p.tiles * kGrBlock;
  // unit -> channel block, first position
  auto locate_unit = [&p](int u, int& cb, int& base) {
    uint32_t q, r;
    gr_divmod((uint32_t)u, (uint32_t)p.k_blocks, p.mg_kb, q, r);
    cb = (int)r;
    base = (int)q * p.span;
  };
  // boxes of a unit's operand: number of the first (counted from one image before the first) and how many; the first one's position
  auto operand = [&p](int base, int& first_chunk, int& chunks) -> int {
    const uint32_t lo = (uint32_t)(base + p.off_min + p.img_pos);
    uint32_t q0, q1, r0, r1;
    gr_divmod(lo, (uint32_t)p.chunk_pos, p.mg_chunk, q0, r0);
    gr_divmod(lo + (uint32_t)(p.span + p.reach - 1), (uint32_t)p.chunk_pos, p.mg_chunk, q1, r1);
    first_chunk = (int)q0;
    chunks = (int)(q1 - q0) + 1;
    return base + p.off_min - (int)r0;
  };

  if (warp == 0) {
    // ------------------------------------------------------------ dL/dO
    if (ptx::elect_one()) {
      const int per_img = p.img_pos / p.chunk_pos;
      int st = 0;
      uint32_t ph = 1u;
      for (int u = first; u < p.units; u += step) {
        int cb, base, c0, chunks;
        locate_unit(u, cb, base);
        operand(base, c0, chunks);
        if (!ptx::mbar_wait<kIdleWaitNs>(&a_empty[st], ph, err, 0x100u + st)) break;
        ptx::mbar_arrive_expect_tx(&raw_full[st], (uint32_t)(chunks * p.chunk_pos * 128));
        int img = c0 / per_img, k = c0 - img * per_img;
        for (int c = 0; c < chunks; ++c) {
          // (columns and rows past an image's, and images that do not exist, arrive as zeros)
          ptx::tma_load_4d(sA + st * p.a_bytes + c * p.chunk_pos * 128, &tmA, &raw_full[st], cb * kGrBlock, 0, k * p.chunk_rows, img - 1);
          if (++k == per_img) { k = 0; ++img; }
        }
        if (++st == p.a_stages) { st = 0; ph ^= 1u; }
      }
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------ filters
    if (ptx::elect_one()) {
      int st = 0;
      uint32_t ph = 1u;
      for (int u = first; u < p.units; u += step) {
        int cb, base;
        locate_unit(u, cb, base);
        if (!ptx::mbar_wait<kIdleWaitNs>(&w_empty[st], ph, err, 0x180u + st)) break;
        ptx::mbar_arrive_expect_tx(&w_full[st], (uint32_t)p.w_bytes);
        for (int t = 0; t < p.taps; ++t)
          ptx::tma_load_2d(sW + st * p.w_bytes + t * p.w_tap_bytes, &tmW, &w_full[st], p.tap_filter[t] * p.gw, cb * kGrBlock);
        if (++st == 2) { st = 0; ph ^= 1u; }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (the whole warp walks the loops, one lane issues)
    const bool leader = ptx::elect_one();
    const uint32_t tmem_base = __shfl_sync(0xFFFFFFFFu, tmem_base_any, 0);
    // 128 x gw x 16: fp32 accumulators, A K-major, B MN-major
    const uint32_t idesc = ((1u << 4) | (p.f16 ? 0u : kIdescBf16Operands) | (1u << 16) | ((uint32_t)(p.gw >> 3) << 17) | ((128u >> 4) << 24));
    const uint64_t adesc0 = ptx::make_smem_desc(0, 16, 1024, 2);
    // a row of W is one output channel's gw input channels: 32 bytes (32-byte swizzle, code 6) or 64 (code 4)
    const uint64_t bdesc0 = ptx::make_smem_desc(0, 16, 16u * (uint32_t)p.gw, p.gw == 16 ? 6u : 4u);
    const uint32_t a_hi = (uint32_t)(adesc0 >> 32), b_hi = (uint32_t)(bdesc0 >> 32);
    const uint32_t a_lo0 = (uint32_t)adesc0 + (ptx::smem_u32(sA) >> 4), b_lo0 = (uint32_t)bdesc0 + (ptx::smem_u32(sW) >> 4);
    const uint32_t b_step = 2u * (uint32_t)p.gw;  // 16 rows of W, in 16-byte units
    // a group of 32 channels is two MMAs (K slices) on the same columns
    const uint32_t tap16 = (uint32_t)(p.w_tap_bytes >> 4);
    const uint32_t wide = p.gw == 32 ? 1u : 0u, d1 = p.gw == 32 ? 0u : 16u;
    auto wait_all = [&](uint64_t* bar, uint32_t parity, unsigned int code) -> bool {
      return __all_sync(0xFFFFFFFFu, ptx::mbar_wait(bar, parity, err, code));
    };
    // All MMAs of a unit: TILES accumulators per class, SLICES of 16 channels. Both are constants, so that the loop over the taps holds nothing
    // but descriptor words and MMAs (with tests in it an MMA took 125 clocks, without them 51).
    auto issue_unit = [&](auto tiles_tag, auto slices_tag, uint32_t a_st, uint32_t b_st, uint32_t d0) {
      constexpr int TILES = decltype(tiles_tag)::value, SLICES = decltype(slices_tag)::value;
      uint32_t b_t = b_st;
      for (int cls = 0, t = 0; cls < p.classes; ++cls) {
        uint32_t accumulate = 0u;
        const uint32_t d_c = d0 + (uint32_t)(cls * TILES * kGrBlock);
        for (; t < p.class_end[cls]; ++t, b_t += tap16) {
          const uint32_t a_t = a_st + (uint32_t)p.tap_off[t] * 8u;
          if (leader) {
#pragma unroll
            for (int k = 0; k < TILES; ++k) {
              // MMA q: channels 16 q .. of the block, 32 bytes along the row of A, 16 rows further in W; to the columns of its group
#pragma unroll
              for (int q = 0; q < SLICES; ++q)
                ptx::mma_f16_ss(d_c + (uint32_t)(k * kGrBlock) + (q & 2 ? 32u : 0u) + (q & 1 ? d1 : 0u),
                                ((uint64_t)a_hi << 32) | (a_t + (uint32_t)(k * 1024 + 2 * q)), ((uint64_t)b_hi << 32) | (b_t + b_step * (uint32_t)q),
                                idesc, q & 1 ? accumulate | wide : accumulate);
            }
          }
          accumulate = 1u;
        }
      }
    };
    int ast = 0, wst = 0, acc = 0;
    uint32_t aph = 0, wph = 0, cph = 1u;
    for (int u = first; u < p.units; u += step) {
      int cb, base;
      locate_unit(u, cb, base);
      const int left = p.C - cb * kGrBlock, slices = (left < kGrBlock ? left : kGrBlock) >> 4;  // MMAs (16 channels each) of a tap and tile
      if (!wait_all(&acc_empty[acc], cph, 0x200u + acc)) break;
      if (!wait_all(&w_full[wst], wph, 0x380u + wst)) break;
      if (!wait_all(&a_full[ast], aph, 0x300u + ast)) break;
      ptx::tc_fence_after_sync();
      const uint32_t d0 = tmem_base + (uint32_t)(acc * acc_cols);
      int c0, chunks;
      const uint32_t a_st = a_lo0 + (uint32_t)(ast * (p.a_bytes >> 4) + (base + p.off_min - operand(base, c0, chunks)) * 8);
      const uint32_t b_st = b_lo0 + (uint32_t)(wst * (p.w_bytes >> 4));
      auto with_tiles = [&](auto slices_tag) {
        if (p.tiles == 1) issue_unit(std::integral_constant<int, 1>{}, slices_tag, a_st, b_st, d0);
        else if (p.tiles == 2) issue_unit(std::integral_constant<int, 2>{}, slices_tag, a_st, b_st, d0);
        else if (p.tiles == 3) issue_unit(std::integral_constant<int, 3>{}, slices_tag, a_st, b_st, d0);
        else issue_unit(std::integral_constant<int, 4>{}, slices_tag, a_st, b_st, d0);
      };
      if (slices == 4) with_tiles(std::integral_constant<int, 4>{});
      else if (slices == 3) with_tiles(std::integral_constant<int, 3>{});
      else if (slices == 2) with_tiles(std::integral_constant<int, 2>{});
      else with_tiles(std::integral_constant<int, 1>{});
      if (leader) {
        ptx::tc_commit(&a_empty[ast]);
        ptx::tc_commit(&w_empty[wst]);
        ptx::tc_commit(&acc_full[acc]);
      }
      if (++ast == p.a_stages) { ast = 0; aph ^= 1u; }
      if (++wst == 2) { wst = 0; wph ^= 1u; }
      if (++acc == 2) { acc = 0; cph ^= 1u; }
    }
  } else if (warp >= 4 && warp < 8) {
    // ------------------------------------------------------------ epilogue
    const int q = warp & 3;
    int acc = 0;
    uint32_t cph = 0;
    for (int u = first; u < p.units; u += step) {
      int cb, base;
      locate_unit(u, cb, base);
      const int end = base + p.span < p.len ? base + p.span : p.len;
      if (!__all_sync(0xFFFFFFFFu, ptx::mbar_wait<kIdleWaitNs>(&acc_full[acc], cph, err, 0x600u + acc))) break;
      ptx::tc_fence_after_sync();
      for (int k = 0; k < p.tiles; ++k) {
        const int L = base + k * 128 + q * 32 + lane;
        uint32_t img, h, w;
        gr_locate(p, (uint32_t)L, img, h, w);
        for (int cls = 0; cls < p.classes; ++cls) {
          const int hh = (int)h * p.stride + (cls >> 1), ww = (int)w * p.stride + (cls & 1);
          const bool inside = L < end && hh < p.H && ww < p.W;
          uint8_t* dst = inside ? p.dD + ((((int64_t)img * p.H + hh) * p.W + ww) * p.C + cb * kGrBlock) * 2 : nullptr;
          const bool last = k + 1 == p.tiles && cls + 1 == p.classes;
          store_rows<kGrBlock>(tmem_base_any + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * acc_cols + (cls * p.tiles + k) * kGrBlock), dst,
                               p.C - cb * kGrBlock, p.aligned32 != 0, nullptr, last ? &acc_empty[acc] : nullptr, F16 || p.f16 != 0);
        }
      }
      if (++acc == 2) { acc = 0; cph ^= 1u; }
    }
  } else {
    // ------------------------------------------------------------ pruner
    // A group of 8 positions x 4 pairs of vectors is one pass of a warp (a quarter of a warp reads or writes 8 different 16-byte columns: no
    // bank conflicts). Positions of padding hold zeros, which prune to zeros.
    const int pw = warp == 3 ? 0 : warp - 7;  // 0 .. 16
    const int row8 = lane >> 2, pair = lane & 3;
    uint8_t* mine = sA + row8 * 128;
    const int chunk_a = ((2 * pair) ^ row8) * 16, chunk_b = ((2 * pair + 1) ^ row8) * 16;
    with_pattern(p.m, p.n, [&](auto m_tag, auto n_tag) {
      constexpr int M = decltype(m_tag)::value;
      constexpr int N = decltype(n_tag)::value;
      int st = 0;
      uint32_t ph = 0;
      for (int u = first; u < p.units; u += step) {
        int cb, base, c0, chunks;
        locate_unit(u, cb, base);
        const int start = operand(base, c0, chunks);
        const int groups = (chunks * p.chunk_pos + 7) >> 3;
        if (!__all_sync(0xFFFFFFFFu, ptx::mbar_wait(&raw_full[st], ph, err, 0x900u + st))) break;
#pragma unroll 1
        for (int g = pw; g < groups; g += kGrPruneWarps) {
          uint8_t* row = mine + st * p.a_bytes + g * 1024;
          uint4 wa = *(const uint4*)(row + chunk_a), wb = *(const uint4*)(row + chunk_b);
          int64_t num = 0;  // number of the first vector in dO (random keys; any value where there is no vector)
          if (SCHEME == SDGP_RANDOM) {
            uint32_t img, h, x;
            const int L = start + 8 * g + row8;
            gr_locate(p, (uint32_t)(L < 0 ? 0 : L), img, h, x);
            num = (((int64_t)img * p.P + h) * p.Q + x) * (p.C >> 3) + cb * 8 + 2 * pair;
          }
          prune_dense_pair<M, N, SCHEME, F16>(wa, wb, num, p.seed_lo, p.seed_hi, pair & 1);
          *(uint4*)(row + chunk_a) = wa;
          *(uint4*)(row + chunk_b) = wb;
        }
        ptx::fence_proxy_async_smem();  // the tensor core reads through the async proxy
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&a_full[st]);
        if (++st == p.a_stages) { st = 0; ph ^= 1u; }
      }
    });
  }

  __syncwarp();
  if (*(volatile unsigned int*)err != 0u) {
    const uint64_t t0 = ptx::globaltimer_ns();
    while (ptx::globaltimer_ns() - t0 < 200000ull) {
    }
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx::tc_fence_after_sync();
  if (warp == 1) ptx::tmem_dealloc(tmem_base_any, kTmemCols);
}

template <int SCHEME, bool F16>
sdgp_status launch_grouped_scheme(const CUtensorMap& tmA, const CUtensorMap& tmW, const GroupedParams& p, int smem_bytes, cudaStream_t stream) {
  static bool configured[kMaxDevices] = {};
  auto kernel = grouped_fused_kernel<SCHEME, F16>;
  if (!configure_once(kernel, configured)) return SDGP_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(p.units < sm_count() ? p.units : sm_count()));
  cfg.blockDim = dim3(kGrThreads);
  cfg.dynamicSmemBytes = (size_t)(smem_bytes > kSmemAlone ? smem_bytes : kSmemAlone);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, tmA, tmW, p) == cudaSuccess ? SDGP_OK : SDGP_ERR_CUDA;
}

uint32_t gr_magic(int d) { return d <= 1 ? 0xFFFFFFFFu : (uint32_t)(0x100000000ull / (uint64_t)d); }

// Raster, taps and shared memory for `tiles` accumulators a unit and class. False: no plan.
bool plan_grouped(GroupedParams* p, int R, int S, int pad, int tiles, int* smem_bytes) {
  const int stride = p->stride;
  p->classes = stride * stride;
  p->tiles = tiles;
  if (2 * p->classes * tiles * kGrBlock > (int)kTmemCols || R * S > kGrMaxTaps) return false;
  // tap (r, s) of output parity (ph, pw): the pixel of dO it reads lies (ph + pad - r) / stride rows further on
  int most = 0;  // furthest a tap reaches past an image's edge, in either direction of either axis
  for (int c = 0; c < stride; ++c)
    for (int k = (c + pad) % stride; k < (R > S ? R : S); k += stride) {
      const int d = (c + pad - k) / stride;
      most = most > (d < 0 ? -d : d) ? most : (d < 0 ? -d : d);
    }
  const int out_h = (p->H + stride - 1) / stride, out_w = (p->W + stride - 1) / stride;
  p->pitch = (p->Q > out_w ? p->Q : out_w) + most;
  const int64_t img_pos = (int64_t)((p->P > out_h ? p->P : out_h) + most) * p->pitch, len = img_pos * p->B;
  if (len > 0x3FFFFFFF) return false;
  p->img_pos = (int)img_pos;
  p->len = (int)len;
  int lo = 0, hi = 0, t = 0, off[kGrMaxTaps];
  for (int c = 0; c < p->classes; ++c) {
    const int ph = c / stride, pw = c % stride, begin = t;
    for (int r = (ph + pad) % stride; r < R; r += stride)
      for (int s = (pw + pad) % stride; s < S; s += stride) {
        off[t] = (ph + pad - r) / stride * p->pitch + (pw + pad - s) / stride;
        p->tap_filter[t] = (short)(r * S + s);
        lo = t == 0 || off[t] < lo ? off[t] : lo;
        hi = t == 0 || off[t] > hi ? off[t] : hi;
        ++t;
      }
    if (t == begin) return false;  // a parity that no tap reaches: its pixels would have to be cleared
    p->class_end[c] = t;
  }
  p->taps = t;
  p->off_min = lo;
  if (hi - lo > 4096) return false;
  for (int k = 0; k < t; ++k) p->tap_off[k] = (short)(off[k] - lo);
  p->k_blocks = (p->C + kGrBlock - 1) / kGrBlock;
  // Ranges of the line: as few as fit the accumulators, then as many more (shorter ones) as the same number of rounds of units takes.
  const int64_t sms = sm_count(), fewest = (len + 128 * tiles - 1) / (128 * tiles);
  const int64_t rounds = (fewest * p->k_blocks + sms - 1) / sms, ranges = rounds * sms / p->k_blocks;
  p->span = (int)((len + ranges - 1) / ranges);
  const int64_t units = (len + p->span - 1) / p->span * p->k_blocks;
  if (units > 0x3FFFFFFF) return false;
  p->units = (int)units;
  p->reach = hi - lo;
  // Boxes: whole rows of an image, a divisor of its rows so that every box starts where the line has it, some 32 positions (a unit's
  // operand is rounded out to whole boxes)
  const int img_rows = p->img_pos / p->pitch;
  p->chunk_rows = 1;
  for (int d = 2; d <= img_rows && d * p->pitch <= 32; ++d)
    if (img_rows % d == 0) p->chunk_rows = d;
  p->chunk_pos = p->chunk_rows * p->pitch;
  if (p->pitch > 256) return false;
  p->mg_chunk = gr_magic(p->chunk_pos);
  p->mg_pitch = gr_magic(p->pitch);
  p->mg_img = gr_magic(p->img_pos);
  p->mg_kb = gr_magic(p->k_blocks);
  // (the accumulators' rows past the span are not stored, but the tensor core reads their operand)
  const int covered = (p->chunk_pos - 1 + p->span + p->reach + p->chunk_pos - 1) / p->chunk_pos * p->chunk_pos;
  const int read = p->chunk_pos - 1 + 128 * tiles + p->reach;
  p->a_bytes = round_up(covered > read ? covered : read, 8) * 128;
  p->w_tap_bytes = kGrBlock * p->gw * 2;
  p->w_bytes = t * p->w_tap_bytes;
  p->a_stages = (kSmemLimit - 2048 - 2 * p->w_bytes) / p->a_bytes;
  if (p->a_stages < 2) return false;
  if (p->a_stages > kGrMaxStages) p->a_stages = kGrMaxStages;
  p->off_w = p->a_stages * p->a_bytes;
  p->off_bar = p->off_w + 2 * p->w_bytes;
  *smem_bytes = p->off_bar + 1024 + 1024;
  return *smem_bytes <= kSmemLimit;
}

// Estimated time of a plan, us. MMAs and pruning overlap but for a third of the shorter one; every unit has a fixed part, the first unit's pruning
// and the last one's stores are in nobody's shadow. A pruning pass is 8 positions of 64 channels; an MMA takes 16 channels (the last block may
// have fewer than four). Constants fitted to 330 layers of stride 1; over 1088 others within 12 % for nine in ten.
double estimate_grouped(const GroupedParams& p, int m, int scheme) {
  const double pass = scheme == SDGP_MAGNITUDE ? (m == 4 ? 48.0 : 70.0) : scheme == SDGP_RANDOM ? (m == 4 ? 112.0 : 132.0) : (m == 4 ? 100.0 : 105.0);
  const double mma = 53.0 * (p.C / 16.0 / p.k_blocks) * p.taps * p.tiles, prune = (p.span + p.reach + p.chunk_pos) / 8.0 * pass;
  const double longer = mma > prune ? mma : prune, shorter = mma > prune ? prune : mma;
  const int sms = sm_count(), rounds = (p.units + sms - 1) / sms;
  return (rounds * (longer + 0.36 * shorter + 805.0) + prune + 1700.0 * p.tiles * p.classes) / 1900.0 + 2.3;
}

// The fastest plan, if there is one and the call should take it. Stride 2 always does: 488 layers drawn, wide images among them, take 0.52 x the time in
// the mean; seven are 6 to 15 % slower, most wider than 130 pixels, where most others still gain, and neither estimates nor the reach told
// them apart (25 x 15 x 175, 8 groups, 2 x 2, 12.0 us and 13.9; 1 x 57 x 198, 26 groups of 32, 17.1 and 16.8). At stride 1 the other path can be the faster one: every unit prunes its halo anew, so that filters and images with a long reach in
// the line (tall filters, wide images) prune a position two to five times, and filters of 16 taps and more are bound by the MMAs of one group
// each. The rule compares the two estimates: of 1088 layers drawn, tall and wide filters and images among them, 124 are more than 5 % slower here, up
// to 2.7 x; the rule leaves 6 of these, up to 1.15 x, and sends 24 to the other path that were more than 5 % faster here (mean 0.4 % behind the best). Us, the other path and this: 5 x 76 x 76 images,
// 26 groups of 16, 7 x 1, random 2:4, 31.1 and 75.5; 12 x 75 x 144, 15 groups, 3 x 3, random, 68.1 and 105.4; 237 x 16 x 16, 5 groups, 5 x 5,
// random, 31.3 and 40.0; 256 x 14 x 14, 10 groups, 3 x 3, rescaled, 30.1 and 21.9.
bool choose_grouped(int B, int H, int W, int C, int groups, int R, int S, int stride, int pad, const FusedPrune& prune, GroupedParams* best,
                    int* best_smem) {
  const int gw = C / groups;
  if ((gw != 16 && gw != 32) || (int64_t)R * S > kGrMaxTaps || prune.n > 2) return false;
  double best_cost = 0.0;
  *best_smem = 0;
  for (int tiles = 1; tiles <= 4; ++tiles) {
    GroupedParams p = {};
    int smem = 0;
    p.B = B; p.H = H; p.W = W; p.C = C; p.gw = gw; p.stride = stride;
    p.P = (H + 2 * pad - R) / stride + 1;
    p.Q = (W + 2 * pad - S) / stride + 1;
    if (!plan_grouped(&p, R, S, pad, tiles, &smem)) continue;
    // Clocks: 55 an MMA, 130 (magnitude 65) a pruning pass of 8 positions - the longer of the two counts - and 500 between units
    const double mma = 4.0 * 55.0 * p.taps * tiles, prune_clk = (p.span + p.reach + p.chunk_pos) / 8.0 * (prune.scheme == SDGP_MAGNITUDE ? 65.0 : 130.0);
    const int sms = sm_count();
    const double cost = (double)((p.units + sms - 1) / sms) * ((mma > prune_clk ? mma : prune_clk) + 500.0) + prune_clk + 1700.0 * tiles * p.classes;
    if (*best_smem == 0 || cost < best_cost) { *best = p; *best_smem = smem; best_cost = cost; }
  }
  return *best_smem != 0 && (stride == 2 || estimate_grouped(*best, prune.m, prune.scheme) < estimate_block_diagonal(B, H, W, C, groups, R, S, pad, prune));
}

}  // namespace

bool query_grouped(int B, int H, int W, int C, int groups, int R, int S, int stride, int pad, const FusedPrune& prune, int* plan) {
  GroupedParams p;
  int smem;
  if (!choose_grouped(B, H, W, C, groups, R, S, stride, pad, prune, &p, &smem)) return false;
  plan[0] = 1; plan[1] = p.units; plan[2] = p.tiles; plan[3] = p.classes; plan[4] = p.a_stages; plan[5] = p.span;
  return true;
}

sdgp_status launch_grouped_fused(const void* dO, const void* Wg, void* dD, int B, int H, int W, int C, int groups, int R, int S, int stride,
                                 int pad, const FusedPrune& prune, int dtype, cudaStream_t stream) {
  GroupedParams p;
  int best_smem;
  if (!choose_grouped(B, H, W, C, groups, R, S, stride, pad, prune, &p, &best_smem)) return SDGP_ERR_UNSUPPORTED;
  const int gw = p.gw;
  p.dD = (uint8_t*)dD;
  p.n = prune.n; p.m = prune.m;
  p.seed_lo = (uint32_t)prune.seed; p.seed_hi = (uint32_t)(prune.seed >> 32);
  p.f16 = dtype == SDGP_FP16 ? 1 : 0;
  p.aligned32 = ((uintptr_t)dD & 31u) == 0;  // (a pixel's channels are a multiple of 16)
  CUtensorMap tmA, tmW;
  {
    const uint64_t pixel = (uint64_t)C * 2;
    const uint64_t dims[4] = {(uint64_t)C, (uint64_t)p.Q, (uint64_t)p.P, (uint64_t)B};
    const uint64_t strides[3] = {pixel, pixel * p.Q, pixel * p.Q * p.P};
    const uint32_t box[4] = {(uint32_t)kGrBlock, (uint32_t)p.pitch, (uint32_t)p.chunk_rows, 1};
    if (!encode(&tmA, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, dO, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B)) return SDGP_ERR_CUDA;
  }
  {
    const uint64_t cols = (uint64_t)R * S * gw;
    const uint64_t dims[2] = {cols, (uint64_t)C}, strides[1] = {cols * 2};
    const uint32_t box[2] = {(uint32_t)gw, (uint32_t)kGrBlock};
    if (!encode(&tmW, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Wg, dims, strides, box, gw == 16 ? CU_TENSOR_MAP_SWIZZLE_32B : CU_TENSOR_MAP_SWIZZLE_64B))
      return SDGP_ERR_CUDA;
  }
  if (prune.scheme == SDGP_RANDOM) return launch_grouped_scheme<SDGP_RANDOM, false>(tmA, tmW, p, best_smem, stream);
  if (prune.scheme == SDGP_MAGNITUDE) return launch_grouped_scheme<SDGP_MAGNITUDE, false>(tmA, tmW, p, best_smem, stream);
  if (p.f16) return launch_grouped_scheme<SDGP_RESCALED_MAGNITUDE, true>(tmA, tmW, p, best_smem, stream);
  return launch_grouped_scheme<SDGP_RESCALED_MAGNITUDE, false>(tmA, tmW, p, best_smem, stream);
}

cudaError_t take_error_grouped(unsigned int* word) { return take_error_word(word); }

}  // namespace sdgp
