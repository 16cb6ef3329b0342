// The pruning work units of the fused data-gradient kernels.
#pragma once
#include "dgrad_common.cuh"

namespace sdgp {
namespace {

// Fused pruning of four vectors (8 channels each, already in registers) of one pixel row: out[v] = the 8
// compressed bytes of vector v, metaw = their four bytes of position metadata (byte v = the two nibbles of
// vector v). Number of vector v in the whole dL/dO tensor (random keys): vbase + vstep * v. Groups of M = 8, 16
// or 32 channels span 1, 2 or 4 vectors held by neighbouring lanes (lane bits 0 and up; `part` = which of
// them this lane's vectors are); all 32 lanes must call together.
template <int M, int N, int SCHEME, bool F16>
__device__ __forceinline__ void fused_prune_vectors(const uint4 (&w)[4], int64_t vbase, int vstep, uint32_t seed_lo,
                                                    uint32_t seed_hi, int part, uint2 (&out)[4], uint32_t& metaw) {
  uint32_t pos[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    KeepFlags k;
    compress_vector<M, N, SCHEME, F16>(w[v], vbase + vstep * v, seed_lo, seed_hi, part, 0xFFFFFFFFu, out[v], pos[v], k);
  }
  metaw = prmt(prmt(pos[0], pos[1], 0x0073), prmt(pos[2], pos[3], 0x0073), 0x5410);
}

// Four consecutive vectors (numbers vec .. vec + 3, 32 channels) held by one thread: out[t] = the 8 compressed bytes of vector t,
// byte t of metaw = its two position nibbles. Groups of up to 32 stay inside the thread.
template <int M, int N, int SCHEME, bool F16>
__device__ __forceinline__ void fused_prune_quad(const uint4 (&w)[4], int64_t vec, uint32_t seed_lo, uint32_t seed_hi, uint2 (&out)[4],
                                                 uint32_t& metaw) {
  uint32_t pos[4];
  if constexpr (M == 32) {
    compress_quad32<N, SCHEME, F16>(w, vec, seed_lo, seed_hi, out, pos);
  } else {
#pragma unroll
    for (int t = 0; t < 4; t += 2) {
      uint4 pair;
      KeepFlags ka, kb;
      compress_pair<M, N, SCHEME, F16>(w[t], w[t + 1], vec + t, seed_lo, seed_hi, 0, 0u, pair, pos[t], pos[t + 1], ka, kb);
      out[t] = make_uint2(pair.x, pair.y);
      out[t + 1] = make_uint2(pair.z, pair.w);
    }
  }
  metaw = prmt(prmt(pos[0], pos[1], 0x0073), prmt(pos[2], pos[3], 0x0073), 0x5410);
}

// 16 bytes from global memory, read-only path, kept out of L1 (each byte is used once by this SM).
__device__ __forceinline__ uint4 ldg_stream(const uint8_t* ptr) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(ptr));
  return v;
}

// Calls f(group size, n) with the two as compile-time constants.
template <typename F>
__device__ __forceinline__ void with_pattern(int m, int n, F f) {
  using std::integral_constant;
  auto with_n = [&](auto mt) {
    if (n == 1) f(mt, integral_constant<int, 1>{});
    else f(mt, integral_constant<int, 2>{});
  };
  if (m == 4) with_n(integral_constant<int, 4>{});
  else if (m == 8) with_n(integral_constant<int, 8>{});
  else if (m == 16) with_n(integral_constant<int, 16>{});
  else with_n(integral_constant<int, 32>{});
}

}  // namespace
}  // namespace sdgp
