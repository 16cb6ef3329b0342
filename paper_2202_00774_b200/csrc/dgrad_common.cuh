// Shared by the data-gradient kernels: tile and pipeline constants, descriptors, the epilogue, host-side helpers.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>

#include <type_traits>

#include "prune_core.cuh"
#include "ptx.cuh"
#include "sdgp_internal.cuh"

namespace sdgp {

// Where dD goes: element (b, h, w, channel 0) of the launch's output grid is at base + b * sb + h * sh + w * sw (bytes;
// stride-2 convolutions: of one output parity, (0, 0) where a launch holds all four), `channels` elements of 16 bits per pixel (a store is clipped there).
struct OutView {
  uint8_t* base;
  int64_t sw, sh, sb;
  int channels;   // a multiple of 8
  int aligned32;  // base and every pixel start on a 32-byte boundary
};

// Where one launch reads and writes: dO as stored (P x Q pixels of `a_channels` channels per image,
// a multiple of the channel block; W holds only the first `Cout` of them), the full filter
// width in W columns, and the (possibly strided) view of dD the launch fills.
struct DgradView {
  int P, Q, batch;
  int a_channels;                 // channels per pixel of dO that exist
  int meta_channels;              // ... and of the compressed form's metadata rows (whole blocks of 128)
  int64_t w_cols;                 // R_full * S_full * Cin
  OutView d;
};

// Encodes a tiled tensor map, or takes it from the calling thread's cache. False: a driver call failed.
bool encode(CUtensorMap* tm, CUtensorMapDataType dt, int rank, const void* base, const uint64_t* dims, const uint64_t* strides_bytes,
            const uint32_t* box, CUtensorMapSwizzle swz);
// Ordinal of the current device, -1 if it cannot be asked or is not below kMaxDevices.
constexpr int kMaxDevices = 64;
int current_device();

namespace {

// Error word of this translation unit's kernels on each device (read and cleared by take_error_word).
__device__ unsigned int g_device_error = 0;

inline cudaError_t take_error_word(unsigned int* word) {
  cudaError_t e = cudaMemcpyFromSymbol(word, g_device_error, sizeof(*word));
  const unsigned int zero = 0;
  if (e == cudaSuccess && *word != 0) e = cudaMemcpyToSymbol(g_device_error, &zero, sizeof(zero));
  return e;
}

constexpr int kBM = 128;             // output pixels (rows) per CTA tile = TMEM lanes
constexpr int kThreadsGemm = 320;    // 10 warps
constexpr unsigned kIdleWaitNs = 200;  // sleep between polls of the waits that are off the critical path
constexpr int kEHwBytes = kBM * 16;  // rearranged metadata of one (tap, channel block): 128 lanes x 16 B
constexpr int kSlabBytes = 32 * 128;  // epilogue staging of a warp (store_box): 32 rows of 64 columns, once or twice
constexpr uint32_t kTmemCols = 512;
constexpr int kMaxImgRows = 192;     // pixel rows of one A stage (filter-row reuse: TW * (TH + R - 1))
constexpr int kSmemLimit = 232448;   // opt-in dynamic shared memory per CTA
constexpr int kSmemSlack = 1536;     // 1024-byte alignment of the carve + barrier block
// A CTA asks for at least this much, so that no two share a multiprocessor: the second sits in its TMEM allocation until the first is done,
// and the multiprocessor it could have had stays empty (29 x 16 x 16 images, 128 -> 128, dense, tiles of one strip of 64 columns: 19.1 us
// with its pruning pass, 12.3 alone).
constexpr int kSmemAlone = 116 * 1024;
constexpr int kMaxStages = 8;


template <bool SPARSE, int BN>
struct Cfg {
  static constexpr int kKB = SPARSE ? 128 : 64;               // W rows (output channels) per MMA group
  static constexpr int kBCols = BN / 2;                       // W columns staged by one CTA
  static constexpr int kBoxCols = kBCols % 64 == 0 ? 64 : 32;  // columns of one W box
  static constexpr int kBoxes = kBCols / kBoxCols;
  static constexpr int kRowB = kBoxCols * 2;                  // bytes of one W row in shared memory
  static constexpr uint32_t kBSwizzle = (kRowB == 128) ? 2u : 4u;  // descriptor code: 128-/64-byte swizzle
  static constexpr int kBoxBytes = kKB * kRowB;
  static constexpr int kTapBBytes = kBoxBytes * kBoxes;       // one CTA's W bytes of one (tap, channel block)
  static_assert(BN % 64 == 0 && BN <= 256, "64-column slabs; at most 256 columns per MMA");
};

// Grouped convolution: input channels n0 .. n0 + BN - 1 belong to groups n0 / cin_g and up, whose output channels
// start at (n0 / cin_g) * cout_g; the tile's window of channel blocks (kbc channels each) starts at that channel's
// block, or at `diag_last` where the window would otherwise run past the last block (W is zero outside the groups'
// own blocks, so a window that covers more than it must changes nothing).
template <class P>
__device__ __forceinline__ int first_k_block(const P& p, int n0, int kbc) {
  if (p.diag_cin_g == 0) return 0;
  const int kb = ((n0 / p.diag_cin_g) * p.diag_cout_g) / kbc;
  return kb < p.diag_last ? kb : p.diag_last;
}

// Instruction descriptor: fp32 accumulate, bf16 A and B, A K-major, B MN-major, M = 256 (pair).
__host__ __device__ constexpr uint32_t make_idesc(int n, bool sparse) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(256 >> 4) << 24) | (sparse ? (1u << 2) : 0u);
}
// The A-format (bits 7-9) and B-format (bits 10-12) fields: 1 = bf16, 0 = binary16. Both operands
// always have the same type.
constexpr uint32_t kIdescBf16Operands = (1u << 7) | (1u << 10);

// Every position nibble of real metadata is at least 4 (p0 | p1 << 2 with p0 < p1), so a 16-bit
// group of four nibbles is at least 0x4444; pixels outside the image arrive as zeros. The
// per-half maximum with 0x4444 therefore leaves real metadata alone and turns a missing group
// into the well-formed position pair (0,1) in every chunk.
__device__ __forceinline__ uint32_t well_formed(uint32_t x) { return __vmaxu2(x, 0x44444444u); }

// 64 columns of the 32 accumulator rows of a warp: TMEM -> registers -> 16-bit pairs. The barriers (null: none) of the MMA thread
// are signalled as soon as the columns are in registers: first_read - they may then hold the next tile's metadata -, released - the
// accumulator has been read to its end.
__device__ __forceinline__ void read_slab(uint32_t taddr, uint32_t (&packed)[32], uint64_t* first_read, uint64_t* released, bool f16) {
  uint32_t v0[32], v1[32];
  ptx::tmem_ld_32x32(taddr, v0);
  ptx::tmem_ld_32x32(taddr + 32u, v1);
  ptx::tmem_ld_wait();
  if (first_read != nullptr || released != nullptr) {
    ptx::tc_fence_before_sync();
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
      if (first_read != nullptr) ptx::mbar_arrive_cluster(first_read, 0);
      if (released != nullptr) ptx::mbar_arrive_cluster(released, 0);
    }
  }
  if (f16) {
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      packed[e] = pack_pair_rn<true>(__uint_as_float(v0[2 * e]), __uint_as_float(v0[2 * e + 1]));
      packed[16 + e] = pack_pair_rn<true>(__uint_as_float(v1[2 * e]), __uint_as_float(v1[2 * e + 1]));
    }
  } else {
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      packed[e] = pack_pair_rn<false>(__uint_as_float(v0[2 * e]), __uint_as_float(v0[2 * e + 1]));
      packed[16 + e] = pack_pair_rn<false>(__uint_as_float(v1[2 * e]), __uint_as_float(v1[2 * e + 1]));
    }
  }
}

// A warp's 32 rows (pixels) of a 128-row x BN accumulator to global memory. The four epilogue warps share nothing: no barrier
// between them and no shared tile (but in store_patch). Against one staging tile for all four, two barriers per slab and one TMA store of the whole
// patch, a small layer ends 1-2 us earlier (256 x 512 . 512 x 256, dense: 7.6 -> 5.8 us per call).
//
// store_rows: straight from registers. Each thread writes whole 32-byte sectors of its own row and L2 puts the lines together; the
// shortest way from an accumulator to memory (702 x 256 . 256 x 192: 7.1 us against 8.5 us through store_box).
// dst: the row's address at the tile's first channel, nullptr if the row lies outside dD; columns: channels of dD left from
// there (warp-uniform). released: the MMA thread's barrier for the accumulator.
template <int BN>
__device__ __forceinline__ void store_rows(uint32_t taddr, uint8_t* dst, int columns, bool aligned32, uint64_t* first_slab_read,
                                           uint64_t* released, bool f16) {
#pragma unroll 1
  for (int c0 = 0; c0 < BN; c0 += 64) {
    const bool last = c0 + 64 >= BN || c0 + 64 >= columns;
    uint32_t packed[32];
    read_slab(taddr + (uint32_t)c0, packed, c0 == 0 ? first_slab_read : nullptr, last ? released : nullptr, f16);
    uint8_t* out = dst + 2 * c0;
    if (dst == nullptr) {
    } else if (aligned32 && columns - c0 >= 64) {
#pragma unroll
      for (int c = 0; c < 4; ++c) ptx::st_global_256(out + 32 * c, &packed[8 * c]);
    } else {
#pragma unroll
      for (int c = 0; c < 8; ++c)
        if (c0 + 8 * c < columns) *(uint4*)(out + 16 * c) = make_uint4(packed[4 * c], packed[4 * c + 1], packed[4 * c + 2], packed[4 * c + 3]);
    }
    if (last) break;
  }
}

// store_box: through 4 KB (twice where there is room: the next slab is packed while the last one is stored) of the warp's own swizzled shared memory and its own TMA store (a box of 32 pixels, clipped at the
// edges of dD): one line per request instead of 32 per instruction. For launches whose epilogues run beside other tiles' work:
// the pruning warps of a fused kernel need the load/store unit (128 -> 128 channels at 28 x 28, batch 256: 47 us against 53 us).
// (c1, c2, c3, c4): coordinates 1.. of the box in dD's map; five: the map has five dimensions.
template <int BN>
__device__ __forceinline__ void store_box(uint32_t taddr, uint8_t* stage, const CUtensorMap* tmD, bool five, int n0, int c1, int c2,
                                          int c3, int c4, bool in_range, int columns, uint64_t* first_slab_read, uint64_t* released,
                                          bool f16, int bufs, uint32_t& chunk) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int c0 = 0; c0 < BN; c0 += 64) {
    const bool last = c0 + 64 >= BN || c0 + 64 >= columns;
    uint32_t packed[32];
    read_slab(taddr + (uint32_t)c0, packed, c0 == 0 ? first_slab_read : nullptr, last ? released : nullptr, f16);
    uint8_t* buf = stage + (bufs == 2 ? chunk & 1u : 0u) * kSlabBytes;
    if (lane == 0) {  // the store that last used this buffer has read it
      if (bufs == 2) ptx::bulk_wait_group_read<1>();
      else ptx::bulk_wait_group_read<0>();
    }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < 8; ++c)
      *(uint4*)(buf + lane * 128 + ((c ^ (lane & 7)) << 4)) =
          make_uint4(packed[4 * c], packed[4 * c + 1], packed[4 * c + 2], packed[4 * c + 3]);
    ptx::fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) {
      if (!in_range) {
      } else if (five) ptx::tma_store_5d(tmD, buf, n0 + c0, c1, c2, c3, c4);
      else ptx::tma_store_4d(tmD, buf, n0 + c0, c1, c2, c3);
      ptx::bulk_commit_group();  // (an empty group where nothing is stored: the waits count groups)
    }
    ++chunk;
    if (last) break;
  }
}

// store_patch: the four warps together, a 128-row slab of 64 columns through one 16 KB tile (twice where there is room) and one TMA box of
// the whole patch, clipped at the edges of dD. Two barriers of the four warps a slab, but a quarter of store_box's requests and of the
// write requests that rows make at L2: for launches whose stores set the pace (plan_halo()).
template <int BN, bool FIVE>
__device__ __forceinline__ void store_patch(uint32_t taddr, uint8_t* staging, int bufs, const CUtensorMap* tmD, int n0, int c1, int c2, int c3,
                                            int c4, bool in_range, uint32_t& chunk, uint64_t* first_slab_read, bool f16) {
  const int row = ((threadIdx.x >> 5) & 3) * 32 + (threadIdx.x & 31);
  const bool issuer = row == 0;
#pragma unroll 1
  for (int c0 = 0; c0 < BN; c0 += 64, ++chunk) {
    uint32_t packed[32];
    read_slab(taddr + (uint32_t)c0, packed, c0 == 0 ? first_slab_read : nullptr, nullptr, f16);
    uint8_t* buf = staging + (bufs == 2 ? chunk & 1u : 0u) * 4 * kSlabBytes;
    if (issuer) {  // the store that last used this buffer has read it
      if (bufs == 2) ptx::bulk_wait_group_read<1>();
      else ptx::bulk_wait_group_read<0>();
    }
    ptx::named_bar_sync(1, 128);
#pragma unroll
    for (int c = 0; c < 8; ++c)
      *(uint4*)(buf + row * 128 + ((c ^ (row & 7)) << 4)) =
          make_uint4(packed[4 * c], packed[4 * c + 1], packed[4 * c + 2], packed[4 * c + 3]);
    ptx::fence_proxy_async_smem();
    ptx::named_bar_sync(1, 128);
    if (issuer) {
      if (!in_range) {
      } else if (FIVE) ptx::tma_store_5d(tmD, buf, n0 + c0, c1, c2, c3, c4);
      else ptx::tma_store_4d(tmD, buf, n0 + c0, c1, c2, c3);
      ptx::bulk_commit_group();  // (an empty group where nothing is stored: the waits count groups)
    }
  }
}

// Opts `kernel` in to the large dynamic shared-memory carve, once per device and instantiation.
template <typename K>
bool configure_once(K kernel, bool (&done)[kMaxDevices]) {
  const int dev = current_device();
  if (dev < 0) return false;
  if (!done[dev]) {
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) != cudaSuccess) return false;
    done[dev] = true;
  }
  return true;
}

inline int round_up(int x, int a) { return (x + a - 1) / a * a; }

// CTA pairs of a persistent grid over `tiles` work items.
inline int pairs_for(int tiles) {
  const int max_pairs = sm_count() / 2;
  return tiles < max_pairs ? tiles : max_pairs;
}

// When a contraction lets the next kernel of its stream be scheduled: as soon as it runs, or (0) only when its CTAs leave. Behind a
// contraction of compressed operands usually comes the next layer's pruning, whose blocks the scheduler deals to the
// multiprocessors that the contraction leaves free, up to eight to each, and there they stay: a small tensor's whole grid then runs on a
// handful of multiprocessors. That is no loss where the contraction leaves about half of the chip. Pooling and ReLU above 2412 x 128
// -> 448 (70 pairs), pruning + contraction: 10.0 us early, 7.3 late; residual above 5684 x 512 -> 512: 19.3, 15.5; 256 images of
// 14 x 14 x 256, 3 x 3: 54.7, 51.2. Contractions followed by contractions (fused, dense) win 1-3 % by the early launch.
inline int early_for(bool before_pruning, int pairs) { return !before_pruning || 2 * pairs * 100 <= 55 * sm_count(); }

// Launch as clusters of two CTAs with programmatic stream serialisation: the grid may be scheduled while the previous kernel
// of the stream drains (the kernel waits for it after its set-up).
template <typename... Params, typename... Args>
sdgp_status launch_pairs(void (*kernel)(Params...), int pairs, int threads, int smem_bytes, cudaStream_t stream, const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(2 * pairs));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = (size_t)(smem_bytes > kSmemAlone ? smem_bytes : kSmemAlone);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, args...) == cudaSuccess ? SDGP_OK : SDGP_ERR_CUDA;
}

}  // namespace
}  // namespace sdgp
