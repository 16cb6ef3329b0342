// N:M pruning of the output data gradient (Algorithm 1, Section 3.2), sm_100a.
//
// A thread owns pairs of aligned runs of 8 elements (a 256-bit load each); where a dense copy is asked for, and below a pooling, single
// runs of 8. Groups of m = 4, 8 and 16 are ranked inside the thread (16: single runs span two lanes); groups of 32 span two lanes
// (four), which trade their keys with warp shuffles. The kernel is a pure stream: 2 B read per element, 1 B of compressed values, 1/8 B of
// position metadata (+ 1/8 B mask, + 2 B dense copy when asked for), every output indexed by the run's number so all stores coalesce.
#include <cuda_bf16.h>

#include "prune_core.cuh"
#include "ptx.cuh"
#include "sdgp_internal.cuh"

namespace sdgp {
namespace {

constexpr int kThreads = 256;
constexpr int kVecPerThread = 4;
// Resident blocks per SM the compiler is asked to make room for. Pruning dL/dO itself under the magnitude function: six
// (40 registers; five measured the same for groups of 4 and 3 % slower for groups of 8). The random and rescaled functions:
// five (48 registers; six spill and measured 1-5 % slower). The producers below a ReLU keep the compiler's own choice.
template <int SCHEME, int SRC>
constexpr int kBlocksPerSm = SRC != 0 ? 0 : SCHEME == SDGP_MAGNITUDE ? 6 : 5;

// Launch with programmatic stream serialisation: the kernel may be scheduled while the previous
// kernel of the stream is still draining; it waits for that kernel before its first load.
template <typename... Params, typename... Args>
cudaError_t launch_after_previous(void (*kernel)(Params...), dim3 grid, dim3 block, cudaStream_t stream, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = 0;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, Params(args)...);
}

// Where the vectors come from: dL/dO itself; the gradient above a ReLU; the gradient above a 2 x 2 max pooling and a ReLU.
enum Source { kPlain, kRelu, kPool };

// The producer of dL/dO below a ReLU (Section 2.1, Fig. 2): the 8 gradients g above the ReLU pass where the
// ReLU's activation a is positive (a number greater than zero: sign clear, magnitude between 1 and the
// pattern of infinity) and become +0.0 elsewhere. nan_add = 0x7FFF - (pattern of infinity) in both half-words:
// adding it to a magnitude sets the half-word's top bit exactly for the NaN patterns.
struct ReluSource {
  const uint4* act;   // the ReLU's activation, same shape as the gradient; nullptr: no ReLU, the input is dL/dO itself
  uint4* grad;        // optional: the unpruned dL/dO (kept for the weight gradient, Section 3.1)
  uint32_t nan_add;
  const uint4* skip;  // optional: the second gradient that reaches the ReLU where a residual connection joins its
                      // branch; the two are added before the gate
  int f16;            // element type of the sum (only read when skip is set)
  // 2 x 2 max pooling of stride 2 above the ReLU (pool_k8 != 0): the input gradient has the pooled shape
  // [B, H/2, W/2, K] and `act` the full one [B, H, W, K]; pool_k8 = K / 8, pool_hp = H / 2, pool_wp = W / 2.
  int pool_k8, pool_hp, pool_wp;
  bool aligned32;     // every vector tensor that is read (and `grad`) starts on a 32-byte boundary
};

// Two 16-bit elements of each gradient, added in fp32 (one rounding) and rounded to the 16-bit type to nearest-even;
// a NaN sum becomes the canonical quiet NaN.
template <bool F16>
__device__ __forceinline__ uint32_t add_pair(uint32_t g, uint32_t s) {
  const float lo = __fadd_rn(lane_lo<F16>(g), lane_lo<F16>(s)), hi = __fadd_rn(lane_hi<F16>(g), lane_hi<F16>(s));
  return f32_to_elem_bits<F16>(lo) | (f32_to_elem_bits<F16>(hi) << 16);
}

__device__ __forceinline__ uint32_t relu_pass2(uint32_t g, uint32_t a, uint32_t nan_add) {
  const uint32_t mag = a & 0x7FFF7FFFu;
  const uint32_t nonzero = mag + 0x7FFF7FFFu, nan = mag + nan_add;   // top bit of each half-word
  const uint32_t ok = nonzero & ~nan & ~a;
  return g & prmt(ok, 0u, 0xBB99);  // top bits replicated over their half-words
}

__device__ __forceinline__ uint4 add_vectors(const uint4& g, const uint4& k, int f16) {
  return f16 ? make_uint4(add_pair<true>(g.x, k.x), add_pair<true>(g.y, k.y), add_pair<true>(g.z, k.z), add_pair<true>(g.w, k.w))
             : make_uint4(add_pair<false>(g.x, k.x), add_pair<false>(g.y, k.y), add_pair<false>(g.z, k.z), add_pair<false>(g.w, k.w));
}

__device__ __forceinline__ uint4 relu_vector(const uint4& g, const uint4& a, uint32_t nan_add) {
  return make_uint4(relu_pass2(g.x, a.x, nan_add), relu_pass2(g.y, a.y, nan_add), relu_pass2(g.z, a.z, nan_add),
                    relu_pass2(g.w, a.w, nan_add));
}

// Vectors v and v + 1 of dL/dO below a ReLU: the gradients above it, wa and wb, plus the second gradient where there is one,
// gated by the activation; written out as well if the caller keeps the unpruned tensor.
__device__ __forceinline__ void relu_pair(int64_t v, bool aligned32, const ReluSource& src, uint4& wa, uint4& wb) {
  uint4 aa, ab;
  load_pair(src.act + v, aligned32, aa, ab);
  if (src.skip) {
    uint4 ka, kb;
    load_pair(src.skip + v, aligned32, ka, kb);
    wa = add_vectors(wa, ka, src.f16);
    wb = add_vectors(wb, kb, src.f16);
  }
  wa = relu_vector(wa, aa, src.nan_add);
  wb = relu_vector(wb, ab, src.nan_add);
  if (src.grad) {
    src.grad[v] = wa;
    src.grad[v + 1] = wb;
  }
}

// Pooling backward for one 32-bit word (two channels) of a window: a[0..3] are the activation words at the window's
// four positions in the order (0,0), (0,1), (1,0), (1,1), g the pooled gradient's word. Per channel the gradient goes
// to the first largest activation if that is a number greater than zero. Both channels at once, in 16-bit lanes:
// key = the pattern where it is a positive number, else 0 (15 bits; patterns of positive numbers order like the
// numbers); (key_a | 0x8000) - key_b keeps the lane's top bit exactly when key_a >= key_b, and no borrow leaves the
// lane. Position t wins when its key is strictly above every earlier one and not below any later one; position 0
// must also be non-zero (a later winner is above a key that is at least zero).
__device__ __forceinline__ void pool_select2(const uint32_t (&a)[4], uint32_t g, uint32_t nan_add, uint32_t (&out)[4]) {
  constexpr uint32_t H = 0x80008000u;
  uint32_t k[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) k[t] = relu_pass2(a[t], a[t], nan_add);
  const uint32_t ge01 = (k[0] | H) - k[1], ge02 = (k[0] | H) - k[2], ge03 = (k[0] | H) - k[3];
  const uint32_t ge12 = (k[1] | H) - k[2], ge13 = (k[1] | H) - k[3], ge23 = (k[2] | H) - k[3];
  const uint32_t nz0 = k[0] + 0x7FFF7FFFu;  // top bit of a lane: its key is not zero
  uint32_t win[4];
  win[0] = (ge01 & ge02 & ge03) & (nz0 & H);
  win[1] = (~ge01 & ge12 & ge13) & H;
  win[2] = (~ge02 & ~ge12 & ge23) & H;
  win[3] = (~ge03 & ~ge13 & ~ge23) & H;
#pragma unroll
  for (int t = 0; t < 4; ++t) out[t] = g & prmt(win[t], 0u, 0xBB99);  // top bits replicated over their half-words
}

// The four vectors a thread prunes and their numbers in dL/dO (>= nvec: none). Without pooling they are the thread's
// slots of four consecutive 256-vector stripes (every load of a warp is one contiguous 512 bytes). With pooling a
// thread owns the four pixels of one window for one 8-channel vector: it reads the pooled gradient once and the four
// activation vectors, and its lanes still hold neighbouring channel vectors of the same pixel.
template <int SRC>
__device__ __forceinline__ void load_unit(const uint4* __restrict__ dO, int64_t nvec, const ReluSource& src,
                                          int64_t (&vi)[kVecPerThread], uint4 (&in)[kVecPerThread]) {
  if (SRC == kPool) {
    const int64_t u = (int64_t)blockIdx.x * kThreads + threadIdx.x;  // number of the pooled gradient's vector
    const bool live = u < (nvec >> 2);
    int64_t pix00 = 0;
    int cv = 0;
    if (live) {  // (the host checked that the number of pooled vectors fits 32 bits)
      const uint32_t window = (uint32_t)u / (uint32_t)src.pool_k8;
      cv = (int)((uint32_t)u - window * (uint32_t)src.pool_k8);
      const uint32_t t = window / (uint32_t)src.pool_wp;
      const uint32_t j = window - t * (uint32_t)src.pool_wp;
      const uint32_t b = t / (uint32_t)src.pool_hp;
      const uint32_t i = t - b * (uint32_t)src.pool_hp;
      pix00 = (((int64_t)b * src.pool_hp * 2 + 2 * i) * src.pool_wp + j) * 2;  // pixel (2i, 2j) of image b
    }
    uint4 a[4];
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      vi[it] = live ? (pix00 + (it >> 1) * (2 * src.pool_wp) + (it & 1)) * src.pool_k8 + cv : nvec;
      a[it] = live ? __ldg(src.act + vi[it]) : make_uint4(0u, 0u, 0u, 0u);
    }
    uint4 g = live ? __ldg(dO + u) : make_uint4(0u, 0u, 0u, 0u);
    if (live && src.skip) {  // a second gradient of the pooled shape (a residual connection joins below the pooling)
      g = add_vectors(g, __ldg(src.skip + u), src.f16);
    }
    uint32_t ox[4], oy[4], oz[4], ow[4];
    const uint32_t ax[4] = {a[0].x, a[1].x, a[2].x, a[3].x}, ay[4] = {a[0].y, a[1].y, a[2].y, a[3].y},
                   az[4] = {a[0].z, a[1].z, a[2].z, a[3].z}, aw[4] = {a[0].w, a[1].w, a[2].w, a[3].w};
    pool_select2(ax, g.x, src.nan_add, ox);
    pool_select2(ay, g.y, src.nan_add, oy);
    pool_select2(az, g.z, src.nan_add, oz);
    pool_select2(aw, g.w, src.nan_add, ow);
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      in[it] = make_uint4(ox[it], oy[it], oz[it], ow[it]);
      if (live && src.grad) src.grad[vi[it]] = in[it];
    }
    return;
  }
  const int64_t base = (int64_t)blockIdx.x * (kThreads * kVecPerThread) + threadIdx.x;
#pragma unroll
  for (int it = 0; it < kVecPerThread; ++it) {
    vi[it] = base + (int64_t)it * kThreads;
    in[it] = make_uint4(0, 0, 0, 0);
    if (vi[it] < nvec) {
      in[it] = __ldg(dO + vi[it]);
      if (SRC == kRelu) {
        if (src.skip) in[it] = add_vectors(in[it], __ldg(src.skip + vi[it]), src.f16);
        in[it] = relu_vector(in[it], __ldg(src.act + vi[it]), src.nan_add);
        if (src.grad) src.grad[vi[it]] = in[it];
      }
    }
  }
}

// Row pitch of the metadata in pairs of vectors (two bytes each): k16 per input row, kpad16 per output row (kpad16 == 0: same as
// the input). A reader that takes rows by TMA needs whole 16-byte rows of metadata; the values need no padding.
struct MetaPitch {
  uint32_t k16, kpad16;
};

// Position of pair p's metadata; the thread that owns a row's last pair names the position pair (0, 1) in the padding.
__device__ __forceinline__ int64_t meta_index(int64_t p, bool fits32, uint16_t* __restrict__ meta, MetaPitch pitch) {
  const int64_t row = fits32 ? (int64_t)((uint32_t)p / pitch.k16) : p / pitch.k16;  // (a 64-bit division is some 80 instructions)
  const uint32_t kp = (uint32_t)(p - row * pitch.k16);
  const int64_t po = row * pitch.kpad16 + kp;
  if (kp == pitch.k16 - 1 && meta)
    for (uint32_t t = 1; t <= pitch.kpad16 - pitch.k16; ++t) meta[po + t] = (uint16_t)0x4444;
  return po;
}

// Keep flags (bit 15 of each lane) as the vector's mask byte, in the TOP byte of the result.
__device__ __forceinline__ uint32_t mask_top_byte(const KeepFlags& k) {
  constexpr uint32_t H = 0x80008000u;
  uint32_t x = k.k0 & H;
  x = (x >> 1) | (k.k1 & H);
  x = (x >> 1) | (k.k2 & H);
  x = (x >> 1) | (k.k3 & H);       // bits 12..15 and 28..31: elements 0..3 of chunk A and of chunk B
  return x * 0x00001001u;          // ... side by side in bits 24..31
}

// Writes one vector's outputs from the lane-paired form (see m4_prune_vector). COMPRESS: every
// 4-chunk holds at most two survivors, so values / meta can be produced.
template <bool COMPRESS>
__device__ __forceinline__ void emit_packed(int64_t v, uint32_t y0, uint32_t y1, uint32_t y2, uint32_t y3,
                                            uint32_t km0, uint32_t km1, uint32_t km2, uint32_t km3,
                                            uint4* __restrict__ dense, uint2* __restrict__ values,
                                            uint8_t* __restrict__ meta, uint8_t* __restrict__ mask) {
  const uint4 pruned = make_uint4(prmt(y0, y1, 0x5410), prmt(y2, y3, 0x5410), prmt(y0, y1, 0x7632), prmt(y2, y3, 0x7632));
  const KeepFlags k = {km0, km1, km2, km3};
  if (dense) dense[v] = pruned;
  if (mask) mask[v] = (uint8_t)(mask_top_byte(k) >> 24);
  if (COMPRESS && (values || meta)) {
    uint2 out, slot_mask;
    uint32_t pos_top;
    gather_slots<false>(pruned, k, out, slot_mask, pos_top);
    if (values) values[v] = out;
    if (meta) meta[v] = (uint8_t)(pos_top >> 24);
  }
}

// Algorithm 1 for m = 4 (any n) and for groups of 8, 16 and 32 with n <= 2. Bound: HBM for the magnitude function of m = 4,
// the integer pipe for the others. Without a dense copy a thread owns PAIRS of vectors: 32-byte loads, 16 bytes of values, two
// of metadata and two of mask per store - half the memory instructions and address arithmetic per element of the
// one-vector form, and a group of 16 needs no shuffles. DENSE (a dense pruned copy is asked for, or n > 2) and the pooling
// source, whose threads own the four pixels of a window, keep single vectors.
template <int M, int N, int SCHEME, bool F16, int SRC, bool DENSE>
__global__ void __launch_bounds__(kThreads, kBlocksPerSm<SCHEME, SRC>)
prune_kernel(const uint4* __restrict__ dO, int64_t nvec, uint32_t seed_lo, uint32_t seed_hi,
             uint4* __restrict__ dense, uint2* __restrict__ values, uint8_t* __restrict__ meta,
             uint8_t* __restrict__ mask, MetaPitch pitch, ReluSource src) {
  ptx::wait_for_previous_grid();
  ptx::launch_dependents();  // only once this grid's own predecessor is done: at most one grid ever waits behind a running one
  if constexpr (!DENSE && SRC != kPool) {
    constexpr int kPairs = kVecPerThread / 2;
    const int64_t npair = nvec >> 1;  // (nvec is even)
    const int64_t base = (int64_t)blockIdx.x * kThreads + threadIdx.x, stride = (int64_t)gridDim.x * kThreads;
    const bool al = src.aligned32;
    uint4 wa[kPairs], wb[kPairs];
#pragma unroll
    for (int it = 0; it < kPairs; ++it) {
      const int64_t p = base + it * stride;
      wa[it] = wb[it] = make_uint4(0u, 0u, 0u, 0u);
      if (p < npair) {
        load_pair(dO + 2 * p, al, wa[it], wb[it]);
        if (SRC == kRelu) relu_pair(2 * p, al, src, wa[it], wb[it]);
      }
    }
#pragma unroll
    for (int it = 0; it < kPairs; ++it) {
      const int64_t p = base + it * stride;
      if (M == 32 ? !__any_sync(0xFFFFFFFFu, p < npair) : p >= npair) continue;  // (the lanes of a group of 32 meet in shuffles)
      uint4 out;
      uint32_t pa, pb;
      KeepFlags ka, kb;
      compress_pair<M, N, SCHEME, F16>(wa[it], wb[it], 2 * p, seed_lo, seed_hi, M == 32 ? (int)(threadIdx.x & 1) : 0, 0xFFFFFFFFu,
                                       out, pa, pb, ka, kb);
      if (M == 32 && p >= npair) continue;
      const int64_t po = pitch.kpad16 == 0 ? p : meta_index(p, npair <= 0xFFFFFFFF, (uint16_t*)meta, pitch);
      if (values) ((uint4*)values)[p] = out;
      if (meta) ((uint16_t*)meta)[po] = (uint16_t)prmt(pa, pb, 0x0073);
      if (mask) ((uint16_t*)mask)[p] = (uint16_t)prmt(mask_top_byte(ka), mask_top_byte(kb), 0x0073);
    }
  } else {
    constexpr int LANES = M <= 8 ? 1 : M / 8;
    const int part = (int)(threadIdx.x & (LANES - 1));
    uint4 in[kVecPerThread];
    int64_t vi[kVecPerThread];
    load_unit<SRC>(dO, nvec, src, vi, in);
#pragma unroll
    for (int it = 0; it < kVecPerThread; ++it) {
      const int64_t v = vi[it];
      if (LANES == 1 && v >= nvec) continue;
      if constexpr (!DENSE) {
        uint2 out;
        uint32_t pos_top;
        KeepFlags k;
        compress_vector<M, N, SCHEME, F16>(in[it], v, seed_lo, seed_hi, part, 0xFFFFFFFFu, out, pos_top, k);
        if (LANES > 1 && v >= nvec) continue;
        if (values) values[v] = out;
        if (meta) meta[v] = (uint8_t)(pos_top >> 24);
        if (mask) mask[v] = (uint8_t)(mask_top_byte(k) >> 24);
      } else {
        uint32_t y0, y1, y2, y3, km0, km1, km2, km3;
        if constexpr (M == 4)
          m4_prune_vector<N, SCHEME, F16>(in[it], v, seed_lo, seed_hi, y0, y1, y2, y3, km0, km1, km2, km3);
        else
          top2_prune_vector<M, SCHEME, F16>(in[it], v, seed_lo, seed_hi, N, part, 0xFFFFFFFFu, y0, y1, y2, y3, km0, km1, km2, km3);
        if (LANES > 1 && v >= nvec) continue;
        emit_packed<(N <= 2)>(v, y0, y1, y2, y3, km0, km1, km2, km3, dense, values, meta, mask);
      }
    }
  }
}

// Only the rescaled scheme reads values as numbers: the other two run the same (bf16-named)
// instantiation for both element types.
template <int M, int N, int SRC>
cudaError_t launch_select(int scheme, bool f16, const void* dO, int64_t nvec, uint64_t seed, void* dense, void* values,
                          void* meta, void* mask, MetaPitch pitch, cudaStream_t stream, ReluSource src) {
  if (nvec == 0) return cudaSuccess;
  const uint32_t lo = (uint32_t)seed, hi = (uint32_t)(seed >> 32);
  auto launch = [&](auto kernel, bool pairs) {
    // Pairs: two per thread, or one where all blocks of that split are resident at once anyway (a small tensor is a matter of
    // latency: 256 x 512 elements take 32 blocks instead of 16; groups of 32, whose lanes wait for each other's keys, gain by it up to a
    // block per multiprocessor only). A warp whose second pairs all lie past the end leaves them out: 1067 x 2112, 2:32 with a mask, 4.8 us
    // when it went through their ranking, 3.0 without. A persistent grid that prefetches a thread's next pair measured 3-15 % slower
    // than blocks that come and go.
    const int64_t singles = (nvec + 2 * kThreads - 1) / (2 * kThreads);
    const int64_t per_block = pairs && singles <= (M == 32 ? 1 : 4) * (int64_t)sm_count() ? 2 * kThreads : kThreads * kVecPerThread;
    const int64_t blocks = (nvec + per_block - 1) / per_block;
    if (blocks > 0x7FFFFFFF) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)blocks), block(kThreads);
    return launch_after_previous(kernel, grid, block, stream, (const uint4*)dO, nvec, lo, hi, (uint4*)dense, (uint2*)values,
                                 (uint8_t*)meta, (uint8_t*)mask, pitch, src);
  };
#define SDGP_SELECT(S, F)                                                                                          \
  if (N > 2 || dense) return launch(prune_kernel<M, N, S, F, SRC, true>, false);                                \
  else if constexpr (N <= 2) return launch(prune_kernel<M, N, S, F, SRC, false>, SRC != kPool)
  if (scheme == SDGP_RANDOM) { SDGP_SELECT(SDGP_RANDOM, false); }
  else if (scheme == SDGP_MAGNITUDE) { SDGP_SELECT(SDGP_MAGNITUDE, false); }
  else if (f16) { SDGP_SELECT(SDGP_RESCALED_MAGNITUDE, true); }
  else { SDGP_SELECT(SDGP_RESCALED_MAGNITUDE, false); }
#undef SDGP_SELECT
}

template <int SRC>
cudaError_t launch_prune_src(const void* dO, int64_t rows, int64_t K, int n, int m, int scheme, uint64_t seed, void* dense,
                             void* values, void* meta, void* mask, cudaStream_t stream, int64_t k_pad, int dtype,
                             ReluSource src) {
  const bool f16 = dtype == SDGP_FP16;
  const int64_t nvec = rows * (K / 8);
  MetaPitch pitch = {(uint32_t)(K / 16), 0};
  if (k_pad != 0 && k_pad != K) {
    // padded metadata rows exist only for compressed outputs
    if (k_pad < K || k_pad % 16 != 0 || K % 16 != 0 || n > 2 || dense || SRC != kPlain) return cudaErrorInvalidValue;
    pitch.kpad16 = (uint32_t)(k_pad / 16);
  }
  switch (m) {
    case 4:
      switch (n) {
        case 1: return launch_select<4, 1, SRC>(scheme, f16, dO, nvec, seed, dense, values, meta, mask, pitch, stream, src);
        case 2: return launch_select<4, 2, SRC>(scheme, f16, dO, nvec, seed, dense, values, meta, mask, pitch, stream, src);
        case 3: return launch_select<4, 3, SRC>(scheme, f16, dO, nvec, seed, dense, values, meta, mask, pitch, stream, src);
        default: return launch_select<4, 4, SRC>(scheme, f16, dO, nvec, seed, dense, values, meta, mask, pitch, stream, src);
      }
#define SDGP_M_CASE(M)                                                                                     \
  case M:                                                                                                  \
    if (n == 1) return launch_select<M, 1, SRC>(scheme, f16, dO, nvec, seed, dense, values, meta, mask, pitch, stream, src); \
    if (n == 2) return launch_select<M, 2, SRC>(scheme, f16, dO, nvec, seed, dense, values, meta, mask, pitch, stream, src); \
    if (SRC != kPlain || values || meta) return cudaErrorInvalidValue;                                        \
    return launch_rank(dO, nvec, n, m, scheme, seed, dense, mask, stream, dtype); /* reads dL/dO itself */
    SDGP_M_CASE(8)
    SDGP_M_CASE(16)
    SDGP_M_CASE(32)
#undef SDGP_M_CASE
    default: return cudaErrorInvalidValue;
  }
}

bool aligned32(const void* p) { return ((uintptr_t)p & 31u) == 0; }

}  // namespace

cudaError_t launch_prune(const void* dO, int64_t rows, int64_t K, int n, int m, int scheme,
                         uint64_t seed, void* dense, void* values, void* meta, void* mask,
                         cudaStream_t stream, int64_t k_pad, int dtype) {
  return launch_prune_src<kPlain>(dO, rows, K, n, m, scheme, seed, dense, values, meta, mask, stream, k_pad, dtype,
                                  ReluSource{nullptr, nullptr, 0u, nullptr, 0, 0, 0, 0, aligned32(dO)});
}

cudaError_t launch_relu_backward_prune(const void* dY, const void* act, int64_t rows, int64_t K, int n, int m, int scheme,
                                       uint64_t seed, void* grad, void* dense, void* values, void* meta, void* mask,
                                       cudaStream_t stream, int dtype, const void* skip) {
  const ReluSource src = {(const uint4*)act, (uint4*)grad, dtype == SDGP_FP16 ? 0x03FF03FFu : 0x007F007Fu,
                          (const uint4*)skip, dtype == SDGP_FP16 ? 1 : 0, 0, 0, 0,
                          aligned32(dY) && aligned32(act) && aligned32(skip)};
  return launch_prune_src<kRelu>(dY, rows, K, n, m, scheme, seed, dense, values, meta, mask, stream, 0, dtype, src);
}

cudaError_t launch_maxpool_relu_backward_prune(const void* dYp, const void* act, int B, int H, int W, int64_t K, int n, int m,
                                               int scheme, uint64_t seed, void* grad, void* dense, void* values, void* meta,
                                               void* mask, cudaStream_t stream, int dtype, const void* skip_pooled) {
  const ReluSource src = {(const uint4*)act, (uint4*)grad, dtype == SDGP_FP16 ? 0x03FF03FFu : 0x007F007Fu,
                          (const uint4*)skip_pooled, dtype == SDGP_FP16 ? 1 : 0, (int)(K / 8), H / 2, W / 2, false};
  return launch_prune_src<kPool>(dYp, (int64_t)B * H * W, K, n, m, scheme, seed, dense, values, meta, mask, stream, 0, dtype, src);
}

namespace {

// One thread per 8-channel vector of the result: four 128-bit loads, one store. A positive number's pattern orders like the
// number; what is not positive counts as +0 and a NaN (of either sign) above everything. HBM-bound: 2.5 B per element of x.
__global__ void __launch_bounds__(kThreads)
relu_maxpool_kernel(const uint4* __restrict__ x, uint4* __restrict__ y, int64_t nout, int64_t k8, int64_t wp, uint32_t nan_add) {
  const int64_t u = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  if (u >= nout) return;
  const int64_t window = u / k8, c = u - window * k8;
  const int64_t row = window / wp, j = window - row * wp;  // row: pooled row of all images together
  const int64_t v = ((2 * row * wp + j) * 2) * k8 + c;     // x's pixel (2 row, 2 j)
  auto key = [nan_add](uint32_t a) -> uint32_t {
    const uint32_t mag = a & 0x7FFF7FFFu;
    return mag & prmt((mag + nan_add) | ~a, 0u, 0xBB99);  // top bits replicated over their half-words
  };
  uint4 best = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const uint4 a = __ldg(x + v + (t >> 1) * (2 * wp * k8) + (t & 1) * k8);
    best = make_uint4(__vmaxu2(best.x, key(a.x)), __vmaxu2(best.y, key(a.y)), __vmaxu2(best.z, key(a.z)), __vmaxu2(best.w, key(a.w)));
  }
  y[u] = best;
}

}  // namespace

cudaError_t launch_relu_maxpool(const void* x, int64_t B, int64_t H, int64_t W, int64_t K, int dtype, void* y, cudaStream_t stream) {
  const int64_t nout = B * (H / 2) * (W / 2) * (K / 8), blocks = (nout + kThreads - 1) / kThreads;
  if (nout == 0) return cudaSuccess;
  if (blocks > 0x7FFFFFFF) return cudaErrorInvalidValue;
  relu_maxpool_kernel<<<(unsigned)blocks, kThreads, 0, stream>>>((const uint4*)x, (uint4*)y, nout, K / 8, W / 2,
                                                                 dtype == SDGP_FP16 ? 0x03FF03FFu : 0x007F007Fu);
  return cudaGetLastError();
}

}  // namespace sdgp
