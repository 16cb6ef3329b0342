// Fused prune + contraction over rows: dD [rows, N] = prune(dO [rows, K]) . W [K, N], for fully connected layers and 1 x 1
// convolutions (no taps, so no halo and no metadata masters).
//
// What it is for: layers bound by memory or by latency. The two-pass path moves 2 B per element of dO to the prune kernel, 1.125 B
// back to memory and 1.125 B into the contraction; here dO is read once and its compressed form never leaves the SM.
//
// A CTA pair takes 256 rows and a group of up to seven tiles of BN output columns, all of whose accumulators sit in TMEM at once: a
// block of 128 channels is pruned once into a stage of shared memory, meets the W of every column tile of the group, and is gone. With more
// columns than TMEM holds, groups go to neighbouring pairs, which prune the same rows again (their dO comes from L2).
//
// Warp roles (24 warps): warp 0 streams dense dO by TMA (two swizzled boxes of 64 channels per block), warp 2 streams W, warp 1 of
// the pair's first CTA issues the MMAs, warps 4..7 are the epilogue (one per TMEM lane quarter), warps 8..23 prune: each takes 8
// rows of every block, a thread 32 channels of one row - four vectors from shared memory (8 rows of one chunk per load phase: no
// bank conflicts), so that groups of up to 32 never leave the thread, two 16-byte stores of values, two half-words of metadata.
// All addresses are fixed per thread but for the stage. A first version loaded dO from global memory into the pruning warps'
// registers: 117 instructions per vector (64 here), half of them addresses, and 40 % of its warps waiting for loads (1024 -> 256
// channels, 50176 rows: 51 us against 32). What bounds it now: issue slots of the pruning warps, some 1400 clocks per block.
#include "dgrad_prune.cuh"
#include "dgrad_rows.cuh"

namespace sdgp {
namespace {

constexpr int kRowsThreads = 24 * 32;
constexpr int kRowsPruneWarps = 16;
constexpr int kRowsMaxStages = 8;            // of each ring
constexpr int kRowsOutBytes = 4 * 2 * kSlabBytes;  // epilogue staging
constexpr int kRowsMaxAcc = 8;               // accumulators
constexpr int kABytes = 128 * 128;           // 128 rows x 64 compressed elements, 128-byte swizzled
constexpr int kMetaBytes = 128 * 16;         // the stage's metadata in the order tcgen05.cp moves to TMEM
constexpr int kRawBytes = 2 * 128 * 128;     // 128 rows x 128 dense channels as two 128-byte-swizzled boxes

template <int BN, int SCHEME, bool F16>
__global__ void __launch_bounds__(kRowsThreads, 1)
rows_fused_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                  const __grid_constant__ CUtensorMap tmD, const RowsParams p) {
  using C = Cfg<true, BN>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sRaw = smem;
  uint8_t* sA = smem + p.off_a;
  uint8_t* sMeta = smem + p.off_meta;
  uint8_t* sW = smem + p.off_w;
  uint8_t* sOut = smem + p.off_out;
  uint64_t* raw_full = (uint64_t*)(smem + p.off_bar);
  uint64_t* raw_empty = raw_full + kRowsMaxStages;
  uint64_t* a_full = raw_empty + kRowsMaxStages;
  uint64_t* a_empty = a_full + kRowsMaxStages;
  uint64_t* w_ready = a_empty + kRowsMaxStages;
  uint64_t* w_empty = w_ready + kRowsMaxStages;
  uint64_t* acc_full = w_empty + kRowsMaxStages;
  uint64_t* acc_empty = acc_full + kRowsMaxAcc;
  uint32_t* tmem_slot = (uint32_t*)(acc_empty + kRowsMaxAcc);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = ptx::cluster_ctarank();
  unsigned int* err = &g_device_error;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kRowsMaxStages; ++s) {
      ptx::mbar_init(&raw_full[s], 1);
      ptx::mbar_init(&raw_empty[s], kRowsPruneWarps);
      ptx::mbar_init(&a_full[s], 2 * kRowsPruneWarps);  // the pruning warps of both CTAs
      ptx::mbar_init(&a_empty[s], 1);
      ptx::mbar_init(&w_ready[s], 1);
      ptx::mbar_init(&w_empty[s], 1);
    }
    for (int a = 0; a < kRowsMaxAcc; ++a) {
      ptx::mbar_init(&acc_full[a], 1);
      ptx::mbar_init(&acc_empty[a], 8);
    }
    ptx::fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    ptx::prefetch_tensormap(&tmA);
    ptx::prefetch_tensormap(&tmB);
    ptx::prefetch_tensormap(&tmD);
  }
  if (warp == 1) {
    ptx::tmem_alloc_pair(tmem_slot, kTmemCols);
    ptx::tmem_relinquish_pair();
  }
  ptx::tc_fence_before_sync();
  ptx::cluster_sync();
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base_any = *tmem_slot;
  ptx::wait_for_previous_grid();
  ptx::launch_dependents();  // (after every wait without a time limit: see the general kernel)

  const int pair_stride = gridDim.x >> 1;
  const int first_pair = blockIdx.x >> 1;
  const int my_works = first_pair < p.works ? (p.works - first_pair + pair_stride - 1) / pair_stride : 0;
  const int n_half = (int)rank * C::kBCols;
  // work number lt of this CTA: row tile and first / last column tile (the groups of a row tile are neighbours: its rows are in L2)
  auto locate = [&p, first_pair, pair_stride](int lt, int& rt, int& nt0, int& nt1) {
    const int work = first_pair + lt * pair_stride;
    rt = work / p.n_groups;
    nt0 = (work - rt * p.n_groups) * p.group_tiles;
    nt1 = nt0 + p.group_tiles < p.n_tiles ? nt0 + p.group_tiles : p.n_tiles;
  };

  if (warp == 0) {
    // ------------------------------------------------------------ dO producer
    if (ptx::elect_one()) {
      bool alive = true;
      int st = 0;
      uint32_t ph = 1u;
      for (int lt = 0; alive && lt < my_works; ++lt) {
        int rt, nt0, nt1;
        locate(lt, rt, nt0, nt1);
        const int row0 = rt * 256 + (int)rank * 128;
        for (int kb = 0; kb < p.k_blocks; ++kb) {
          if (!ptx::mbar_wait(&raw_empty[st], ph, err, 0x100u + st)) { alive = false; break; }
          ptx::mbar_arrive_expect_tx(&raw_full[st], (uint32_t)kRawBytes);
          ptx::tma_load_2d(sRaw + st * kRawBytes, &tmA, &raw_full[st], kb * 128, row0);
          ptx::tma_load_2d(sRaw + st * kRawBytes + kRawBytes / 2, &tmA, &raw_full[st], kb * 128 + 64, row0);
          if (++st == p.raw_stages) { st = 0; ph ^= 1u; }
        }
      }
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------ W producer
    if (ptx::elect_one()) {
      bool alive = true;
      int st = 0;
      uint32_t ph = 1u;
      for (int lt = 0; alive && lt < my_works; ++lt) {
        int rt, nt0, nt1;
        locate(lt, rt, nt0, nt1);
        for (int kb = 0; alive && kb < p.k_blocks; ++kb) {
          for (int nt = nt0; nt < nt1; ++nt) {
            if (!ptx::mbar_wait(&w_empty[st], ph, err, 0x180u + st)) { alive = false; break; }
            if (rank == 0) ptx::mbar_arrive_expect_tx(&w_ready[st], 2u * (uint32_t)C::kTapBBytes);
#pragma unroll
            for (int j = 0; j < C::kBoxes; ++j)
              ptx::tma_load_2d_pair(sW + st * C::kTapBBytes + j * C::kBoxBytes, &tmB, &w_ready[st], nt * BN + n_half + C::kBoxCols * j,
                                    kb * C::kKB);
            if (++st == p.w_stages) { st = 0; ph ^= 1u; }
          }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------- MMA issuer (first CTA only; the whole warp walks the loops, one lane issues)
    if (rank == 0) {
      const bool leader = ptx::elect_one();
      const uint32_t tmem_base = __shfl_sync(0xFFFFFFFFu, tmem_base_any, 0);
      const uint32_t idesc = make_idesc(BN, true) & ~(p.f16 ? kIdescBf16Operands : 0u);
      const uint64_t adesc0 = ptx::make_smem_desc(0, 16, 1024, 2);
      const uint64_t bdesc0 = ptx::make_smem_desc(0, C::kBoxBytes, 8 * C::kRowB, C::kBSwizzle);
      const uint64_t edesc0 = ptx::make_smem_desc(0, 128, 128, 0);
      const uint32_t a_hi = (uint32_t)(adesc0 >> 32), b_hi = (uint32_t)(bdesc0 >> 32), e_hi = (uint32_t)(edesc0 >> 32);
      const uint32_t a_lo0 = (uint32_t)adesc0 + (ptx::smem_u32(sA) >> 4);
      const uint32_t b_lo0 = (uint32_t)bdesc0 + (ptx::smem_u32(sW) >> 4);
      const uint32_t e_lo0 = (uint32_t)edesc0 + (ptx::smem_u32(sMeta) >> 4);
      constexpr uint32_t kBStep = (uint32_t)((C::kKB / 4) * C::kRowB / 16);
      auto wait_all = [&](uint64_t* bar, uint32_t parity, unsigned int code) -> bool {
        return __all_sync(0xFFFFFFFFu, ptx::mbar_wait(bar, parity, err, code));
      };
      bool alive = true;
      int ast = 0, wst = 0, acc0 = 0;
      uint32_t aph = 0, wph = 0;
      uint32_t acc_ph = 0;  // bit a: phase of accumulator a
      for (int lt = 0; alive && lt < my_works; ++lt) {
        int rt, nt0, nt1;
        locate(lt, rt, nt0, nt1);
        for (int kb = 0; alive && kb < p.k_blocks; ++kb) {
          if (!wait_all(&a_full[ast], aph, 0x300u + ast)) { alive = false; break; }
          const uint32_t e_col = tmem_base + (uint32_t)(p.meta_col + 4 * ast);
          const uint32_t a_lo = a_lo0 + (uint32_t)(ast * (kABytes / 16));
          const int mmas = kb == p.k_blocks - 1 ? p.last_mmas : 4;
          ptx::tc_fence_after_sync();
          if (leader) ptx::tc_cp_128x128b_pair(e_col, ((uint64_t)e_hi << 32) | (e_lo0 + (uint32_t)(ast * (kMetaBytes / 16))));
          for (int nt = nt0; nt < nt1; ++nt) {
            const int acc = acc0 + nt - nt0 < p.acc_ring ? acc0 + nt - nt0 : acc0 + nt - nt0 - p.acc_ring;
            if (kb == 0 && !wait_all(&acc_empty[acc], ((acc_ph >> acc) & 1u) ^ 1u, 0x200u + acc)) { alive = false; break; }
            if (!wait_all(&w_ready[wst], wph, 0x380u + wst)) { alive = false; break; }
            ptx::tc_fence_after_sync();
            if (leader) {
              const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN), b_lo = b_lo0 + (uint32_t)(wst * (C::kTapBBytes / 16));
#pragma unroll
              for (int q = 0; q < 4; ++q)
                if (q < mmas)
                  ptx::mma_sp_f16_ss_pair(d_tmem, ((uint64_t)a_hi << 32) | (a_lo + (uint32_t)(q * 2)),
                                          ((uint64_t)b_hi << 32) | (b_lo + (uint32_t)q * kBStep), e_col + (uint32_t)(q & 2),
                                          idesc | (uint32_t)(q & 1), (kb == 0 && q == 0) ? 0u : 1u);
              ptx::tc_commit_pair(&w_empty[wst], 3);
              if (kb == p.k_blocks - 1) ptx::tc_commit_pair(&acc_full[acc], 3);
            }
            if (++wst == p.w_stages) { wst = 0; wph ^= 1u; }
          }
          if (alive && leader) ptx::tc_commit_pair(&a_empty[ast], 3);
          if (++ast == p.a_stages) { ast = 0; aph ^= 1u; }
        }
        for (int nt = nt0; nt < nt1; ++nt) {
          acc_ph ^= 1u << acc0;
          if (++acc0 == p.acc_ring) acc0 = 0;
        }
      }
    }
  } else if (warp >= 8) {
    // ------------------------------------------------------------ pruner
    const int pw = warp - 8;
    const int r = lane & 7, cg = lane >> 3;  // row of the warp's eight, 32-channel quarter of the block
    const int i = pw * 8 + r;                // row of the tile
    // dense vectors 4 cg .. 4 cg + 3 of the row: box cg / 2, 16-byte chunks 4 (cg % 2) + t, swizzled by the row
    const uint8_t* src = sRaw + (cg >> 1) * (kRawBytes / 2) + i * 128;
    const int chunk0 = 4 * (cg & 1);
    // compressed: chunks 2 cg, 2 cg + 1 of the row; metadata of MMA cg, half h: half-word i / 8 % 2 of line i % 8 + 8 h + 16 (i / 16)
    uint8_t* dst0 = sA + i * 128 + ((2 * cg) ^ r) * 16;
    uint8_t* dst1 = sA + i * 128 + ((2 * cg + 1) ^ r) * 16;
    uint8_t* mdst = sMeta + (r + 16 * (i >> 4)) * 16 + 4 * cg + 2 * ((i >> 3) & 1);
    const int total = my_works * p.k_blocks;
    with_pattern(p.m, p.n, [&](auto m_tag, auto n_tag) {
      constexpr int M = decltype(m_tag)::value;
      constexpr int N = decltype(n_tag)::value;
      int rst = 0, ast = 0, lt = 0, kb = 0;
      uint32_t rph = 0, aph = 1u;
      int64_t vec = 0;  // number of the thread's first vector in dO (random keys)
      uint4 w[4];
      auto load = [&]() -> bool {
        if (!__all_sync(0xFFFFFFFFu, ptx::mbar_wait(&raw_full[rst], rph, err, 0x500u + rst))) return false;
#pragma unroll
        for (int t = 0; t < 4; ++t) w[t] = *(const uint4*)(src + rst * kRawBytes + (((chunk0 + t) ^ r) << 4));
        return true;
      };
      bool alive = total > 0 && load();
      for (int use = 0; alive && use < total; ++use) {
        if (SCHEME == SDGP_RANDOM) {
          if (kb == 0) {
            int rt, nt0, nt1;
            locate(lt, rt, nt0, nt1);
            vec = (int64_t)(rt * 256 + (int)rank * 128 + i) * (p.K >> 3) + 4 * cg;
          }
        }
        uint2 out[4];
        uint32_t metaw;
        fused_prune_quad<M, N, SCHEME, F16>(w, vec + kb * 16, p.seed_lo, p.seed_hi, out, metaw);
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&raw_empty[rst]);
        if (++rst == p.raw_stages) { rst = 0; rph ^= 1u; }
        // the next block's vectors are on their way while this one's results are stored and announced
        if (use + 1 < total) alive = load();
        if (!__all_sync(0xFFFFFFFFu, ptx::mbar_wait(&a_empty[ast], aph, err, 0x900u + ast))) break;
        *(uint4*)(dst0 + ast * kABytes) = make_uint4(out[0].x, out[0].y, out[1].x, out[1].y);
        *(uint4*)(dst1 + ast * kABytes) = make_uint4(out[2].x, out[2].y, out[3].x, out[3].y);
        *(uint16_t*)(mdst + ast * kMetaBytes) = (uint16_t)metaw;
        *(uint16_t*)(mdst + ast * kMetaBytes + 128) = (uint16_t)(metaw >> 16);
        ptx::fence_proxy_async_smem();  // the tensor core reads A and metadata through the async proxy
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive_cluster(&a_full[ast], 0);
        if (++ast == p.a_stages) { ast = 0; aph ^= 1u; }
        if (++kb == p.k_blocks) { kb = 0; ++lt; }
      }
    });
  } else if (warp >= 4) {
    // ------------------------------------------------------------ epilogue
    const int q = warp & 3;
    int acc = 0;
    uint32_t acc_ph = 0, chunk = 0;
    bool alive = true;
    for (int lt = 0; alive && lt < my_works; ++lt) {
      int rt, nt0, nt1;
      locate(lt, rt, nt0, nt1);
      const int row = rt * 256 + (int)rank * 128 + 32 * q;
      for (int nt = nt0; nt < nt1; ++nt) {
        if (!ptx::mbar_wait<kIdleWaitNs>(&acc_full[acc], (acc_ph >> acc) & 1u, err, 0x600u + acc)) { alive = false; break; }
        ptx::tc_fence_after_sync();
        store_box<BN>(tmem_base_any + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN), sOut + q * 2 * kSlabBytes, &tmD, false, nt * BN, row,
                      0, 0, 0, row < p.rows, p.N - nt * BN, nullptr, &acc_empty[acc], p.f16 != 0, 2, chunk);
        acc_ph ^= 1u << acc;
        if (++acc == p.acc_ring) acc = 0;
      }
    }
    if (lane == 0) ptx::bulk_wait_group_read<0>();
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
  if (warp == 1) ptx::tmem_dealloc_pair(tmem_base_any, kTmemCols);
}

template <int BN, int SCHEME, bool F16>
sdgp_status launch_rows_bn(const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmD, const RowsParams& p,
                           cudaStream_t stream) {
  static bool configured[kMaxDevices] = {};
  auto kernel = rows_fused_kernel<BN, SCHEME, F16>;
  if (!configure_once(kernel, configured)) return SDGP_ERR_CUDA;
  return launch_pairs(kernel, pairs_for(p.works), kRowsThreads, p.smem_bytes, stream, tmA, tmB, tmD, p);
}

template <int SCHEME, bool F16>
sdgp_status launch_rows_scheme(int bn, const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmD, const RowsParams& p,
                               cudaStream_t stream) {
  switch (bn) {
    case 64: return launch_rows_bn<64, SCHEME, F16>(tmA, tmB, tmD, p, stream);
    case 128: return launch_rows_bn<128, SCHEME, F16>(tmA, tmB, tmD, p, stream);
    default: return launch_rows_bn<192, SCHEME, F16>(tmA, tmB, tmD, p, stream);
  }
}

// Shared-memory plan: the rings grow in turn while they fit.
bool plan_rows_smem(RowsParams* p, int bn) {
  const int w_bytes = 128 * bn;  // one CTA's half of a W stage
  const int budget = kSmemLimit - kSmemSlack - kRowsOutBytes - 2048;
  int raw = 2, a = 2, w = 2;
  auto used = [&]() { return raw * kRawBytes + a * (kABytes + kMetaBytes) + w * w_bytes; };
  if (used() > budget) return false;
  for (bool grown = true; grown;) {
    grown = false;
    int* const rings[3] = {&w, &raw, &a};
    const int most[3] = {kRowsMaxStages, p->works > sm_count() / 2 || p->k_blocks > 5 ? 5 : p->k_blocks < 2 ? 2 : p->k_blocks, 4};
    for (int k = 0; k < 3; ++k) {
      if (*rings[k] >= most[k]) continue;
      ++*rings[k];
      if (used() > budget) --*rings[k];
      else grown = true;
    }
  }
  p->raw_stages = raw; p->a_stages = a; p->w_stages = w;
  p->off_a = raw * kRawBytes;
  p->off_meta = p->off_a + a * kABytes;
  p->off_w = round_up(p->off_meta + a * kMetaBytes, 1024);
  p->off_out = p->off_w + w * w_bytes;
  p->off_bar = p->off_out + kRowsOutBytes;
  p->smem_bytes = p->off_bar + 1024 + 1024;
  return p->smem_bytes <= kSmemLimit;
}

}  // namespace

namespace {

RowsPlan make_plan(int64_t rows, int K, int N, int stage_clk) {
  RowsPlan best = {};
  if (rows < 1 || rows > 0x7FFFFF00 || K % 8 != 0 || N % 8 != 0) return best;
  const int64_t pairs = sm_count() / 2, row_tiles = (rows + 255) / 256;
  for (int bn = 64; bn <= 192; bn += 64) {
    const int n_tiles = (N + bn - 1) / bn;
    for (int g = 1; g <= n_tiles && g * bn <= 448; ++g) {
      RowsParams p = {};
      p.rows = (int)rows; p.K = K; p.N = N;
      p.k_blocks = (K + 127) / 128;
      p.last_mmas = (K - (p.k_blocks - 1) * 128 + 31) / 32;
      p.n_tiles = n_tiles;
      p.n_groups = (n_tiles + g - 1) / g;
      p.group_tiles = (n_tiles + p.n_groups - 1) / p.n_groups;
      if (p.group_tiles != g || row_tiles * p.n_groups > 0x3FFFFFFF) continue;
      p.works = (int)(row_tiles * p.n_groups);
      p.acc_ring = ((int)kTmemCols - 16) / bn;  // (at most four A stages, four metadata columns each)
      p.meta_col = p.acc_ring * bn;
      if (!plan_rows_smem(&p, bn)) continue;
      // clocks of a work: bytes from memory (a pair's share; fewer pairs at work share more), bytes from L2, shared memory (dO in and
      // out, compressed rows in, W in, both operands read per column tile, the epilogue's staging), pruning, epilogue - whichever
      // is longest, a part of the shared-memory time beside it, and the part of the epilogue that the next work's accumulators wait for
      const double kb = p.k_blocks, busy = p.works < pairs ? (double)p.works / pairs : 1.0;
      const double rate = 20.0 / busy < 55.0 ? 20.0 / busy : 55.0;
      const double mem = (256.0 * K / p.n_groups + 256.0 * g * bn) / rate, l2 = (256.0 * K + 128.0 * kb * g * bn) / 55.0;
      const double smem = (kb * (2.0 * 32768 + 18432 + 128.0 * bn * g + g * 4.0 * (4096 + 16.0 * bn)) + 512.0 * bn * g) / 115.0;
      const double prune = kb * stage_clk + 500.0, out = 16.0 * g * bn;
      double work = mem > l2 ? mem : l2;
      if (smem > work) work = smem;
      if (prune > work) work = prune;
      if (out > work) work = out;
      work += 0.4 * smem;
      if (p.acc_ring < 2 * g) work += 4.0 * bn * (2 * g - p.acc_ring);
      const double rounds = (double)((p.works + pairs - 1) / pairs);
      const double cost = rounds * work + out + 4000.0;
      if (!best.ok || cost < best.cost) best = {true, bn, cost, p};
    }
  }
  return best;
}

}  // namespace

RowsPlan plan_rows(int64_t rows, int K, int N, int stage_clk) {
  struct Entry { int64_t rows; int K, N, stage_clk, sms; RowsPlan plan; };
  constexpr int kEntries = 32;
  static thread_local Entry cache[kEntries] = {};
  static thread_local int next = 0;
  const int sms = sm_count();
  for (const Entry& e : cache)
    if (e.rows == rows && e.K == K && e.N == N && e.stage_clk == stage_clk && e.sms == sms) return e.plan;
  Entry& e = cache[next];
  next = (next + 1) % kEntries;
  e = {rows, K, N, stage_clk, sms, make_plan(rows, K, N, stage_clk)};
  return e.plan;
}

sdgp_status launch_rows_fused(const RowsPlan& plan, const void* dO, const void* W, int w_rows, int w_cols, void* dD,
                              const FusedPrune& prune, int dtype, cudaStream_t stream) {
  RowsParams p = plan.p;
  p.n = prune.n; p.m = prune.m;
  p.seed_lo = (uint32_t)prune.seed; p.seed_hi = (uint32_t)(prune.seed >> 32);
  p.f16 = dtype == SDGP_FP16 ? 1 : 0;
  const int box_cols = (plan.bn / 2) % 64 == 0 ? 64 : 32;
  CUtensorMap tmA, tmB, tmD;
  {
    const uint64_t dims[2] = {(uint64_t)p.K, (uint64_t)p.rows}, strides[1] = {(uint64_t)p.K * 2};
    const uint32_t box[2] = {64, 128};
    if (!encode(&tmA, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, dO, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B)) return SDGP_ERR_CUDA;
  }
  {
    const uint64_t dims[2] = {(uint64_t)w_cols, (uint64_t)w_rows}, strides[1] = {(uint64_t)w_cols * 2};
    const uint32_t box[2] = {(uint32_t)box_cols, 128};
    if (!encode(&tmB, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, W, dims, strides, box,
                box_cols == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B))
      return SDGP_ERR_CUDA;
  }
  {
    const uint64_t pitch = (uint64_t)p.N * 2;
    const uint64_t dims[4] = {(uint64_t)p.N, (uint64_t)p.rows, 1, 1}, strides[3] = {pitch, pitch * p.rows, pitch * p.rows};
    const uint32_t box[4] = {64, 32, 1, 1};
    if (!encode(&tmD, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, dD, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B)) return SDGP_ERR_CUDA;
  }
  if (prune.scheme == SDGP_RANDOM) return launch_rows_scheme<SDGP_RANDOM, false>(plan.bn, tmA, tmB, tmD, p, stream);
  if (prune.scheme == SDGP_MAGNITUDE) return launch_rows_scheme<SDGP_MAGNITUDE, false>(plan.bn, tmA, tmB, tmD, p, stream);
  if (p.f16) return launch_rows_scheme<SDGP_RESCALED_MAGNITUDE, true>(plan.bn, tmA, tmB, tmD, p, stream);
  return launch_rows_scheme<SDGP_RESCALED_MAGNITUDE, false>(plan.bn, tmA, tmB, tmD, p, stream);
}

cudaError_t take_error_rows(unsigned int* word) { return take_error_word(word); }

}  // namespace sdgp
