// Algorithm 1 for patterns that keep more than two elements of groups of 8, 16 or 32 (Section 4.2: 4:8, 8:16, 4:32, 16:32
// ...): a dense pruned copy and / or the keep mask. No compressed form exists for these (a 4-chunk may keep more than two).
//
// Ranking every element against every other of its group by 32-bit comparisons costs m - 1 comparisons and additions per
// element: 67 us (4:8) to 228 us (16:32) for a 134 MB tensor whose traffic takes 42 us. Two selections replace it:
//   m = 8       all 28 comparisons of a group, two groups per register (16-bit lanes), one subtraction each; the seven
//               outcomes of an element are added by carry-save logic (bit 15 of the lanes is the only bit that counts) and the
//               3-bit number of wins is compared with 8 - n: about 9 integer instructions per element.
//   m = 16, 32  bit-sliced radix selection: a thread holds 32 consecutive elements, transposes them into bit planes (bit i
//               of plane b = bit b of element i) and fixes the group's n-th largest key bit by bit with one population
//               count per bit and group, then per bit of the position among equal keys (lower position first): the work per
//               element falls with the group size, about 12 (m = 16) and 9 (m = 32) instructions.
#include "prune_core.cuh"
#include "sdgp_internal.cuh"

namespace sdgp {
namespace {

constexpr int kThreads = 256;
constexpr int kVecPerThread = 4;  // 8-element vectors

__device__ __forceinline__ void store_pair(uint4* ptr, bool aligned32, const uint4& a, const uint4& b) {
  if (aligned32) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(ptr), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w),
                 "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
                 : "memory");
  } else {
    ptr[0] = a;
    ptr[1] = b;
  }
}

// Per-lane a >= b (bit 15 of each 16-bit lane; other bits: anything). FULL: 16-bit keys, else 15-bit ones (bit 15 clear).
template <bool FULL>
__device__ __forceinline__ uint32_t lanes_ge(uint32_t a, uint32_t b) {
  constexpr uint32_t H = 0x80008000u;
  if (!FULL) return (a | H) - b;
  const uint32_t t = (a | H) - (b & ~H);
  return lop3<0xB2>(a, b, t);  // (a & ~b) | (~(a ^ b) & t)
}

// ---- groups of 8: the two groups of a pair of vectors in the lanes of eight registers ----
template <int SCHEME, bool F16>
__global__ void __launch_bounds__(kThreads)
rank8_kernel(const uint4* __restrict__ dO, int64_t npair, int n, uint32_t seed_lo, uint32_t seed_hi, uint4* __restrict__ dense,
             uint16_t* __restrict__ mask, bool aligned32) {
  constexpr uint32_t H = 0x80008000u;
  constexpr int kPairs = kVecPerThread / 2;
  const int need = 8 - n;  // wins an element must have at least
  const uint32_t t0 = (need & 1) ? ~0u : 0u, t1 = (need & 2) ? ~0u : 0u, t2 = (need & 4) ? ~0u : 0u;
  const int64_t base = (int64_t)blockIdx.x * (kThreads * kPairs) + threadIdx.x;
  uint4 wa[kPairs], wb[kPairs];
#pragma unroll
  for (int it = 0; it < kPairs; ++it) {
    const int64_t p = base + (int64_t)it * kThreads;
    if (p < npair) load_pair(dO + 2 * p, aligned32, wa[it], wb[it]);
  }
#pragma unroll
  for (int it = 0; it < kPairs; ++it) {
    const int64_t p = base + (int64_t)it * kThreads;
    if (p >= npair) continue;
    uint32_t key[8];  // element i of vector a (low lane) and of vector b; larger ranks first
    {
      uint4 ka = wa[it], kb = wb[it];
      if (SCHEME == SDGP_RANDOM) {
        ka = philox4x32_10((uint32_t)(2 * p), (uint32_t)((uint64_t)(2 * p) >> 32), 0u, 0u, seed_lo, seed_hi);
        kb = philox4x32_10((uint32_t)(2 * p + 1), (uint32_t)((uint64_t)(2 * p + 1) >> 32), 0u, 0u, seed_lo, seed_hi);
      }
      const uint32_t A[4] = {ka.x, ka.y, ka.z, ka.w}, B[4] = {kb.x, kb.y, kb.z, kb.w};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        key[i] = prmt(A[i >> 1], B[i >> 1], (i & 1) ? 0x7632 : 0x5410);
        key[i] = SCHEME == SDGP_RANDOM ? ~key[i] : key[i] & ~H;
      }
    }
    // ge[i][j], i < j: element i beats element j (ties to the lower index); element j beats i iff not
    uint32_t ge[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = i + 1; j < 8; ++j) ge[i][j] = lanes_ge<SCHEME == SDGP_RANDOM>(key[i], key[j]);
    uint32_t km[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      uint32_t w[7];  // outcomes against the other seven
#pragma unroll
      for (int o = 0; o < 7; ++o) {
        const int j = o < i ? o : o + 1;
        w[o] = j > i ? ge[i][j] : ~ge[j][i];  // (the complement folds into the logic operation that reads it)
      }
      const uint32_t s1 = w[0] ^ w[1] ^ w[2], c1 = majority(w[0], w[1], w[2]);
      const uint32_t s2 = w[3] ^ w[4] ^ w[5], c2 = majority(w[3], w[4], w[5]);
      const uint32_t b0 = s1 ^ s2 ^ w[6], c3 = majority(s1, s2, w[6]);
      const uint32_t b1 = c1 ^ c2 ^ c3, b2 = majority(c1, c2, c3);
      // wins < need: the borrow of wins - need
      const uint32_t borrow = majority(~b2, t2, majority(~b1, t1, ~b0 & t0));
      km[i] = prmt(~borrow, 0u, 0xBB99);
    }
    if (mask) {
      uint32_t flags = 0u;
#pragma unroll
      for (int i = 0; i < 8; ++i) flags = (flags >> 1) | (km[i] & H);
      mask[p] = (uint16_t)prmt(flags, 0u, 0x0031);  // bits 8..15: vector a, bits 24..31: vector b
    }
    if (dense) {
      uint32_t ma[4], mb[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        ma[q] = prmt(km[2 * q], km[2 * q + 1], 0x5410);
        mb[q] = prmt(km[2 * q], km[2 * q + 1], 0x7632);
      }
      uint4 ya = make_uint4(wa[it].x & ma[0], wa[it].y & ma[1], wa[it].z & ma[2], wa[it].w & ma[3]);
      uint4 yb = make_uint4(wb[it].x & mb[0], wb[it].y & mb[1], wb[it].z & mb[2], wb[it].w & mb[3]);
      if (SCHEME == SDGP_RESCALED_MAGNITUDE && n < 8) {  // n == m: nothing pruned, nothing rescaled
        auto rescale = [](uint4& y, const uint4& w, const uint32_t (&m)[4]) {
          const float t = __fadd_rn(__fadd_rn(pair_abs<F16>(w.x), pair_abs<F16>(w.y)), __fadd_rn(pair_abs<F16>(w.z), pair_abs<F16>(w.w)));
          const float s = __fadd_rn(__fadd_rn(pair_abs<F16>(y.x), pair_abs<F16>(y.y)), __fadd_rn(pair_abs<F16>(y.z), pair_abs<F16>(y.w)));
          const float sc = s == 0.0f ? 1.0f : __fdiv_rn(t, s);
          const bool finite = is_finite(t);
          y = make_uint4(rescale_slots<F16>(y.x, sc, finite, m[0]), rescale_slots<F16>(y.y, sc, finite, m[1]),
                         rescale_slots<F16>(y.z, sc, finite, m[2]), rescale_slots<F16>(y.w, sc, finite, m[3]));
        };
        rescale(ya, wa[it], ma);
        rescale(yb, wb[it], mb);
      }
      store_pair(dense + 2 * p, aligned32, ya, yb);
    }
  }
}

// ---- groups of 16 and 32: 32 consecutive elements per thread, as 16 words of two ----

// 16 x 16 bit transpose of the low half-words and of the high half-words: bit j of half h of x[b] becomes bit b of half h of
// the old x[j].
__device__ __forceinline__ void transpose16(uint32_t (&x)[16]) {
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const uint32_t a = x[k], b = x[k + 8];
    x[k] = prmt(a, b, 0x6240);
    x[k + 8] = prmt(a, b, 0x7351);
  }
#pragma unroll
  for (int s = 4; s >= 1; s >>= 1) {
    const uint32_t m = s == 4 ? 0x0F0F0F0Fu : s == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      if (k & s) continue;
      const uint32_t a = x[k], b = x[k + s];
      x[k] = (a & m) | ((b << s) & ~m);
      x[k + s] = ((a >> s) & m) | (b & ~m);
    }
  }
}

// One step of the selection for one group: `cand` = elements not yet decided, `need` of them are still to be kept (at least
// one, at most all). Those of `first` (a subset) rank before the rest.
__device__ __forceinline__ void select_step(uint32_t first, uint32_t& cand, uint32_t& keep, int& need) {
  const int c = __popc(first);
  if (c >= need) {
    cand = first;
  } else {
    keep |= first;
    cand ^= first;
    need -= c;
  }
}

template <int M, int SCHEME, bool F16>
__global__ void __launch_bounds__(kThreads)
rank_sliced_kernel(const uint4* __restrict__ dO, int64_t nvec, int n, uint32_t seed_lo, uint32_t seed_hi, uint4* __restrict__ dense,
                   uint32_t* __restrict__ mask, bool aligned32) {
  static_assert(M == 16 || M == 32, "");
  constexpr int G = 32 / M;  // groups of this thread
  const int64_t v = ((int64_t)blockIdx.x * kThreads + threadIdx.x) * kVecPerThread;
  if (v >= nvec) return;
  const bool whole = v + 4 <= nvec;  // (groups of 16: the last thread may have two vectors only)
  uint32_t w[16];
  {
    uint4 q[4];
    q[2] = q[3] = make_uint4(0u, 0u, 0u, 0u);
    load_pair(dO + v, aligned32, q[0], q[1]);
    if (whole) load_pair(dO + v + 2, aligned32, q[2], q[3]);
#pragma unroll
    for (int i = 0; i < 4; ++i) { w[4 * i] = q[i].x; w[4 * i + 1] = q[i].y; w[4 * i + 2] = q[i].z; w[4 * i + 3] = q[i].w; }
  }
  uint32_t plane[16];  // plane[b]: bit j = bit b of element 2j's key, bit 16 + j = of element 2j + 1's; larger keys rank first
  if (SCHEME == SDGP_RANDOM) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint4 o = philox4x32_10((uint32_t)(v + i), (uint32_t)((uint64_t)(v + i) >> 32), 0u, 0u, seed_lo, seed_hi);
      plane[4 * i] = ~o.x; plane[4 * i + 1] = ~o.y; plane[4 * i + 2] = ~o.z; plane[4 * i + 3] = ~o.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i) plane[i] = w[i];
  }
  transpose16(plane);
  uint32_t cand[2] = {G == 1 ? 0xFFFFFFFFu : 0x00FF00FFu, 0xFF00FF00u}, keep[2] = {0u, 0u};
  int need[2] = {n, n};
#pragma unroll
  for (int b = SCHEME == SDGP_RANDOM ? 15 : 14; b >= 0; --b)  // (magnitudes: the sign plane is not looked at)
#pragma unroll
    for (int g = 0; g < G; ++g) select_step(cand[g] & plane[b], cand[g], keep[g], need[g]);
  // equal keys: lower position first, one bit of the position at a time
#pragma unroll
  for (int b = M == 32 ? 4 : 3; b >= 0; --b) {
    const uint32_t low = b == 4 ? 0x00FF00FFu : b == 3 ? 0x0F0F0F0Fu : b == 2 ? 0x33333333u : b == 1 ? 0x55555555u : 0x0000FFFFu;
#pragma unroll
    for (int g = 0; g < G; ++g) select_step(cand[g] & low, cand[g], keep[g], need[g]);
  }
  uint32_t kept = keep[0] | cand[0];
  if (G == 2) kept |= keep[1] | cand[1];

  if (mask) {  // even elements in the low half, odd ones in the high half: interleave
    uint32_t x = kept, t;
    t = (x ^ (x >> 8)) & 0x0000FF00u; x ^= t ^ (t << 8);
    t = (x ^ (x >> 4)) & 0x00F000F0u; x ^= t ^ (t << 4);
    t = (x ^ (x >> 2)) & 0x0C0C0C0Cu; x ^= t ^ (t << 2);
    t = (x ^ (x >> 1)) & 0x22222222u; x ^= t ^ (t << 1);
    mask[v >> 2] = x;  // (a mask is asked for only where rows are whole groups of 32)
  }
  if (!dense) return;
  uint32_t y[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) y[j] = w[j] & prmt(kept << (15 - j), 0u, 0xBB99);  // bits j and 16 + j over their half-words
  if (SCHEME == SDGP_RESCALED_MAGNITUDE && n < M) {
    float t[16], s[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) { t[j] = pair_abs<F16>(w[j]); s[j] = pair_abs<F16>(y[j]); }
#pragma unroll
    for (int width = 16; width > G; width >>= 1)  // balanced pairwise sums in index order
#pragma unroll
      for (int j = 0; j < width / 2; ++j) { t[j] = __fadd_rn(t[2 * j], t[2 * j + 1]); s[j] = __fadd_rn(s[2 * j], s[2 * j + 1]); }
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const float sc = s[g] == 0.0f ? 1.0f : __fdiv_rn(t[g], s[g]);
      const bool finite = is_finite(t[g]);
#pragma unroll
      for (int j = g * (16 / G); j < (g + 1) * (16 / G); ++j)
        y[j] = rescale_slots<F16>(y[j], sc, finite, prmt(kept << (15 - j), 0u, 0xBB99));
    }
  }
  store_pair(dense + v, aligned32, make_uint4(y[0], y[1], y[2], y[3]), make_uint4(y[4], y[5], y[6], y[7]));
  if (whole) store_pair(dense + v + 2, aligned32, make_uint4(y[8], y[9], y[10], y[11]), make_uint4(y[12], y[13], y[14], y[15]));
}

template <int M, int SCHEME, bool F16>
void launch_rank_m(const void* dO, int64_t nvec, int n, uint64_t seed, void* dense, void* mask, cudaStream_t stream) {
  const unsigned blocks = (unsigned)((nvec + kThreads * kVecPerThread - 1) / (kThreads * kVecPerThread));
  const bool aligned32 = (((uintptr_t)dO | (uintptr_t)dense) & 31u) == 0;
  // Plain launches, without programmatic stream serialisation: with it, a stream of back-to-back masked-mode steps (an earlier
  // kernel in this place, dense data-gradient kernel, the same again, ...) once stopped making progress on B200 after a few
  // steps. The cause was not found; the overlap it would buy is small.
  if constexpr (M == 8)
    rank8_kernel<SCHEME, F16><<<blocks, kThreads, 0, stream>>>((const uint4*)dO, nvec >> 1, n, (uint32_t)seed, (uint32_t)(seed >> 32),
                                                               (uint4*)dense, (uint16_t*)mask, aligned32);
  else
    rank_sliced_kernel<M, SCHEME, F16><<<blocks, kThreads, 0, stream>>>((const uint4*)dO, nvec, n, (uint32_t)seed,
                                                                        (uint32_t)(seed >> 32), (uint4*)dense, (uint32_t*)mask, aligned32);
}

template <int M>
void launch_rank_scheme(const void* dO, int64_t nvec, int n, int scheme, uint64_t seed, void* dense, void* mask, cudaStream_t stream,
                        bool f16) {
  if (scheme == SDGP_RANDOM) launch_rank_m<M, SDGP_RANDOM, false>(dO, nvec, n, seed, dense, mask, stream);
  else if (scheme == SDGP_MAGNITUDE) launch_rank_m<M, SDGP_MAGNITUDE, false>(dO, nvec, n, seed, dense, mask, stream);
  else if (f16) launch_rank_m<M, SDGP_RESCALED_MAGNITUDE, true>(dO, nvec, n, seed, dense, mask, stream);
  else launch_rank_m<M, SDGP_RESCALED_MAGNITUDE, false>(dO, nvec, n, seed, dense, mask, stream);
}

}  // namespace

cudaError_t launch_rank(const void* dO, int64_t nvec, int n, int m, int scheme, uint64_t seed, void* dense, void* mask,
                        cudaStream_t stream, int dtype) {
  if (nvec == 0) return cudaSuccess;
  if ((nvec & 1) || (nvec + kThreads * kVecPerThread - 1) / (kThreads * kVecPerThread) > 0x7FFFFFFF) return cudaErrorInvalidValue;
  const bool f16 = dtype == SDGP_FP16;
  if (m == 8) launch_rank_scheme<8>(dO, nvec, n, scheme, seed, dense, mask, stream, f16);
  else if (m == 16) launch_rank_scheme<16>(dO, nvec, n, scheme, seed, dense, mask, stream, f16);
  else if (m == 32) launch_rank_scheme<32>(dO, nvec, n, scheme, seed, dense, mask, stream, f16);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

}  // namespace sdgp
