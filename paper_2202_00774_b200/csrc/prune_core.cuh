// Device code shared by the stand-alone prune kernels and the prune stage fused into the
// data-gradient kernel: the Philox generator, bf16 rounding, packed-lane helpers and the
// per-vector m = 4 pruning function (Algorithm 1, Section 3.2).
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/sdgp.h"

namespace sdgp {
namespace {

// Philox4x32-10 (Salmon et al., SC'11): ten rounds, Weyl key schedule.
__device__ __forceinline__ uint4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                               uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
    const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return make_uint4(c0, c1, c2, c3);
}

// fp32 -> bf16 bits, round to nearest even; any NaN becomes 0x7FC0.
__device__ __forceinline__ uint32_t f32_to_bf16_bits(float f) {
  uint32_t u = __float_as_uint(f);
  if ((u & 0x7FFFFFFFu) > 0x7F800000u) return 0x7FC0u;
  u += 0x7FFFu + ((u >> 16) & 1u);
  return u >> 16;
}

template <int LUT>
__device__ __forceinline__ uint32_t lop3(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(d) : "r"(a), "r"(b), "r"(c), "n"(LUT));
  return d;
}

// prmt.b32, default mode: result byte n = byte (sel nibble n & 7) of {b,a}; a nibble with its
// top bit set replicates that byte's sign bit over the whole result byte instead.
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}

// Truth-table byte of "at least NEED of the three inputs are true", with optional input negation.
template <int NEED>
__host__ __device__ constexpr int threshold_lut(bool na, bool nb, bool nc) {
  int lut = 0;
  for (int idx = 0; idx < 8; ++idx) {
    const int a = ((idx >> 2) & 1) ^ (na ? 1 : 0), b = ((idx >> 1) & 1) ^ (nb ? 1 : 0), c = (idx & 1) ^ (nc ? 1 : 0);
    if (a + b + c >= NEED) lut |= 1 << idx;
  }
  return lut;
}


// 32 bytes of a read-once stream: one 256-bit load where the tensor is 32-byte aligned, else two of 128 bits.
__device__ __forceinline__ void load_pair(const uint4* ptr, bool aligned32, uint4& a, uint4& b) {
  if (aligned32) {
    asm volatile("ld.global.nc.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
                 : "l"(ptr));
  } else {
    a = __ldg(ptr);
    b = __ldg(ptr + 1);
  }
}

// Element type of the 16-bit tensors. Ranking and selection only read bit patterns (the pattern
// with the sign cleared orders bf16 and IEEE binary16 alike); the type matters where the rescale
// of Section 3.2 reads values as numbers and rounds the survivors. F16 = false: bf16, true: binary16.

// fp32 -> binary16 bits, round to nearest even (hardware conversion); any NaN becomes 0x7E00.
__device__ __forceinline__ uint32_t f32_to_f16_bits(float f) {
  const uint32_t h = __half_as_ushort(__float2half_rn(f));
  return ((h & 0x7FFFu) > 0x7C00u) ? 0x7E00u : h;
}

template <bool F16>
__device__ __forceinline__ uint32_t f32_to_elem_bits(float f) {
  return F16 ? f32_to_f16_bits(f) : f32_to_bf16_bits(f);
}

// The element in the low / high half of a lane-paired register as fp32 (exact).
template <bool F16>
__device__ __forceinline__ float lane_lo(uint32_t p) {
  return F16 ? __half2float(__ushort_as_half((unsigned short)(p & 0xFFFFu))) : __uint_as_float(p << 16);
}
template <bool F16>
__device__ __forceinline__ float lane_hi(uint32_t p) {
  return F16 ? __half2float(__ushort_as_half((unsigned short)(p >> 16))) : __uint_as_float(p & 0xFFFF0000u);
}
// ... and their magnitudes
// (the absolute value of the fp32 number clears the same sign bit, NaN payloads included, and rides on the add that
// consumes it instead of costing an integer instruction)
template <bool F16>
__device__ __forceinline__ float lane_lo_abs(uint32_t p) { return fabsf(lane_lo<F16>(p)); }
template <bool F16>
__device__ __forceinline__ float lane_hi_abs(uint32_t p) { return fabsf(lane_hi<F16>(p)); }

// Two fp32 values rounded to nearest even and packed (low, high): hardware conversion, finite inputs.
template <bool F16>
__device__ __forceinline__ uint32_t pack_pair_rn(float lo, float hi) {
  if (F16) {
    const __half2 h = __floats2half2_rn(lo, hi);
    return *(const uint32_t*)&h;
  }
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *(const uint32_t*)&h;
}

// Balanced pairwise sum, in index order, of the magnitudes in the low (high) halves of four
// lane-paired registers: (|e0| + |e1|) + (|e2| + |e3|), every add rounded once.
template <bool F16>
__device__ __forceinline__ float sum4_lo_abs(uint32_t q0, uint32_t q1, uint32_t q2, uint32_t q3) {
  return __fadd_rn(__fadd_rn(lane_lo_abs<F16>(q0), lane_lo_abs<F16>(q1)), __fadd_rn(lane_lo_abs<F16>(q2), lane_lo_abs<F16>(q3)));
}
template <bool F16>
__device__ __forceinline__ float sum4_hi_abs(uint32_t q0, uint32_t q1, uint32_t q2, uint32_t q3) {
  return __fadd_rn(__fadd_rn(lane_hi_abs<F16>(q0), lane_hi_abs<F16>(q1)), __fadd_rn(lane_hi_abs<F16>(q2), lane_hi_abs<F16>(q3)));
}

// Survivors of both lanes times their group's scale, rounded to the element type (nearest even).
// When both group sums are finite every fp32 product is finite and the hardware's packed
// conversion applies (a product beyond the binary16 range rounds to infinity, as IEEE says);
// otherwise (Inf or NaN in the group) each value goes through the explicit rounding, which
// stores any NaN as the one canonical quiet NaN.
template <bool F16>
__device__ __forceinline__ void rescale_packed(uint32_t& y0, uint32_t& y1, uint32_t& y2, uint32_t& y3, uint32_t km0,
                                               uint32_t km1, uint32_t km2, uint32_t km3, float scA, float scB,
                                               float tA, float tB) {
  const bool finite = (__float_as_uint(tA) & 0x7F800000u) != 0x7F800000u &&
                      (__float_as_uint(tB) & 0x7F800000u) != 0x7F800000u;
  if (finite) {
#define SDGP_RESCALE_FAST(y, km) \
  y = pack_pair_rn<F16>(__fmul_rn(lane_lo<F16>(y), scA), __fmul_rn(lane_hi<F16>(y), scB)) & km;
    SDGP_RESCALE_FAST(y0, km0) SDGP_RESCALE_FAST(y1, km1) SDGP_RESCALE_FAST(y2, km2) SDGP_RESCALE_FAST(y3, km3)
#undef SDGP_RESCALE_FAST
  } else {
#define SDGP_RESCALE_SLOW(y, km)                                                 \
  y = (f32_to_elem_bits<F16>(__fmul_rn(lane_lo<F16>(y), scA)) |                  \
       (f32_to_elem_bits<F16>(__fmul_rn(lane_hi<F16>(y), scB)) << 16)) & km;
    SDGP_RESCALE_SLOW(y0, km0) SDGP_RESCALE_SLOW(y1, km1) SDGP_RESCALE_SLOW(y2, km2) SDGP_RESCALE_SLOW(y3, km3)
#undef SDGP_RESCALE_SLOW
  }
}

// The two m = 4 groups of one 8-element vector w (vector number v of the tensor, which fixes the
// random keys). Lane-paired form: register i holds (element i, element i + 4) in its low / high
// 16 bits. Out: y_i = pruned (and, for the rescaled scheme, rescaled) values, km_i = 0xFFFF in
// the lanes of kept elements.
template <int N, int SCHEME, bool F16 = false>
__device__ __forceinline__ void m4_prune_vector(const uint4& w, int64_t v, uint32_t seed_lo, uint32_t seed_hi,
                                                uint32_t& y0, uint32_t& y1, uint32_t& y2, uint32_t& y3,
                                                uint32_t& km0, uint32_t& km1, uint32_t& km2, uint32_t& km3) {
  constexpr int NEED = 4 - N;  // an element is kept iff it beats at least 4 - n of the other three
  // lanes: low half = group A (elements 0..3), high half = group B (elements 4..7)
  const uint32_t p0 = prmt(w.x, w.z, 0x5410), p1 = prmt(w.x, w.z, 0x7632);
  const uint32_t p2 = prmt(w.y, w.w, 0x5410), p3 = prmt(w.y, w.w, 0x7632);

  if (N == 4) {
    km0 = km1 = km2 = km3 = 0xFFFFFFFFu;
  } else if (SCHEME == SDGP_RANDOM) {
    const uint4 o = philox4x32_10((uint32_t)v, (uint32_t)((uint64_t)v >> 32), 0u, 0u, seed_lo, seed_hi);
    // 16-bit keys; smaller ranks first, equal keys: lower index. e(i,j) = r_j - r_i has its
    // sign bit set iff j ranks before i (j < i in key), i.e. iff i loses against j (for i < j).
    const uint32_t rA0 = o.x & 0xFFFFu, rA1 = o.x >> 16, rA2 = o.y & 0xFFFFu, rA3 = o.y >> 16;
    const uint32_t rB0 = o.z & 0xFFFFu, rB1 = o.z >> 16, rB2 = o.w & 0xFFFFu, rB3 = o.w >> 16;
#define SDGP_KEEP4(r0, r1, r2, r3, k0, k1, k2, k3)                                                \
{                                                                                                \
  const uint32_t e01 = r1 - r0, e02 = r2 - r0, e03 = r3 - r0, e12 = r2 - r1, e13 = r3 - r1,      \
                 e23 = r3 - r2;                                                                  \
  k0 = lop3<threshold_lut<NEED>(true, true, true)>(e01, e02, e03);                               \
  k1 = lop3<threshold_lut<NEED>(false, true, true)>(e01, e12, e13);                              \
  k2 = lop3<threshold_lut<NEED>(false, false, true)>(e02, e12, e23);                             \
  k3 = lop3<threshold_lut<NEED>(false, false, false)>(e03, e13, e23);                            \
}
    uint32_t a0, a1, a2, a3, b0, b1, b2, b3;  // keep flags in bit 31
    SDGP_KEEP4(rA0, rA1, rA2, rA3, a0, a1, a2, a3)
    SDGP_KEEP4(rB0, rB1, rB2, rB3, b0, b1, b2, b3)
#undef SDGP_KEEP4
    // replicate the two sign bits over their 16-bit lanes
    km0 = prmt(a0, b0, 0xFFBB); km1 = prmt(a1, b1, 0xFFBB);
    km2 = prmt(a2, b2, 0xFFBB); km3 = prmt(a3, b3, 0xFFBB);
  } else {
    // |x| as 15-bit integers. d(i,j) = (a_i | 0x8000) - a_j per lane never borrows across lanes
    // and has bit 15 of the lane set iff a_i >= a_j, i.e. iff i beats j (i < j: ties to i).
    constexpr uint32_t H = 0x80008000u;
    const uint32_t h0 = p0 | H, h1 = p1 | H, h2 = p2 | H;
    const uint32_t l1 = p1 & ~H, l2 = p2 & ~H, l3 = p3 & ~H;
    const uint32_t d01 = h0 - l1, d02 = h0 - l2, d03 = h0 - l3, d12 = h1 - l2, d13 = h1 - l3, d23 = h2 - l3;
    const uint32_t k0 = lop3<threshold_lut<NEED>(false, false, false)>(d01, d02, d03);
    const uint32_t k1 = lop3<threshold_lut<NEED>(true, false, false)>(d01, d12, d13);
    const uint32_t k2 = lop3<threshold_lut<NEED>(true, true, false)>(d02, d12, d23);
    const uint32_t k3 = lop3<threshold_lut<NEED>(true, true, true)>(d03, d13, d23);
    km0 = prmt(k0, 0, 0xBB99); km1 = prmt(k1, 0, 0xBB99);
    km2 = prmt(k2, 0, 0xBB99); km3 = prmt(k3, 0, 0xBB99);
  }

  y0 = p0 & km0; y1 = p1 & km1; y2 = p2 & km2; y3 = p3 & km3;  // pruned lanes are +0.0
  if (SCHEME == SDGP_RESCALED_MAGNITUDE && N != 4) {
    // per group: scale = sum|x| / sum|kept x|, balanced pairwise sums in index order
    const float tA = sum4_lo_abs<F16>(p0, p1, p2, p3), tB = sum4_hi_abs<F16>(p0, p1, p2, p3);
    const float sA = sum4_lo_abs<F16>(y0, y1, y2, y3), sB = sum4_hi_abs<F16>(y0, y1, y2, y3);
    const float scA = (sA == 0.0f) ? 1.0f : __fdiv_rn(tA, sA);
    const float scB = (sB == 0.0f) ? 1.0f : __fdiv_rn(tB, sB);
    rescale_packed<F16>(y0, y1, y2, y3, km0, km1, km2, km3, scA, scB, tA, tB);
  }

}

// ---- Compressed form of a vector (n <= 2: every 4-chunk keeps at most two elements) ----
//
// A chunk's two slots are two of the four half-words of two registers, so ONE byte permute per chunk gathers them once its
// selector is known, and the position nibbles can be read off that selector. Keep flags live in bit 15 of the two 16-bit
// lanes of a register (low lane: chunk A, elements 0..3; high lane: chunk B, elements 4..7). In flags k0..k3 of a chunk
//   p1 = last survivor, at least 1                  = 1 + [k2 | k3] + [k3]
//   p0 = first survivor if there are two, else 0    = [maj(k1, k2, k3)] + [k2 & k3]
// and a lane of the selector is 0x3210 (p0 = 0, p1 = 1) plus 0x0022 per unit of p0 and 0x2200 per unit of p1 - 1. A byte
// permute in sign-replicating mode turns the flags of both terms into those bytes at once. Against gathering the survivors
// with lane masks (four masks, four ANDs, nine logic operations for slots and positions) this is about half the integer
// instructions of the m = 4 magnitude function (50 -> 30 per vector), which is what bounds the kernels that prune from
// shared memory or registers and the functions with more arithmetic.
struct KeepFlags {
  uint32_t k0, k1, k2, k3;  // bit 15 of each lane: element kept (other bits: anything)
};

__device__ __forceinline__ uint32_t chunk_selectors(uint32_t p0_is_not_0, const KeepFlags& k) {
  const uint32_t two = lop3<0xC0>(k.k2, k.k3, 0u), any = lop3<0xFC>(k.k2, k.k3, 0u);  // k2 & k3, k2 | k3
  // bytes of the result: sign of lane A of the first operand, of lane A of the second, then the same for lane B
  const uint32_t first = prmt(p0_is_not_0, k.k3, 0xFBD9) & 0x22222222u, second = prmt(two, any, 0xFBD9) & 0x22222222u;
  return 0x32103210u + first + second;
}

// Positions p0 | p1 << 2 of chunk A and << 4 of chunk B, in the TOP byte of the result: the four two-bit fields of the
// selectors (bits 1, 9, 17, 25) are brought together by one multiplication (no two partial products share a bit).
__device__ __forceinline__ uint32_t positions_top_byte(uint32_t sel) { return (sel & 0x06060606u) * 0x00820820u; }

__device__ __forceinline__ uint32_t majority(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (c & (a | b)); }

// Keep flags of the two m = 4 groups of a vector under the magnitude or random function (v: number of the vector).
template <int N, int SCHEME>
__device__ __forceinline__ KeepFlags m4_flags(const uint4& w, int64_t v, uint32_t seed_lo, uint32_t seed_hi) {
  constexpr int NEED = 4 - N;  // an element is kept iff it beats at least 4 - n of the other three
  KeepFlags k;
  if (SCHEME == SDGP_RANDOM) {
    const uint4 o = philox4x32_10((uint32_t)v, (uint32_t)((uint64_t)v >> 32), 0u, 0u, seed_lo, seed_hi);
    // 16-bit keys; smaller ranks first, equal keys: lower index. e(i,j) = r_j - r_i has its
    // sign bit set iff j ranks before i (j < i in key), i.e. iff i loses against j (for i < j).
    const uint32_t rA0 = o.x & 0xFFFFu, rA1 = o.x >> 16, rA2 = o.y & 0xFFFFu, rA3 = o.y >> 16;
    const uint32_t rB0 = o.z & 0xFFFFu, rB1 = o.z >> 16, rB2 = o.w & 0xFFFFu, rB3 = o.w >> 16;
    uint32_t a0, a1, a2, a3, b0, b1, b2, b3;  // keep flags in bit 31
#define SDGP_KEEP4(r0, r1, r2, r3, k0, k1, k2, k3)                                                \
{                                                                                                \
  const uint32_t e01 = r1 - r0, e02 = r2 - r0, e03 = r3 - r0,             \
                 e12 = r2 - r1, e13 = r3 - r1, e23 = r3 - r2;            \
  k0 = lop3<threshold_lut<NEED>(true, true, true)>(e01, e02, e03);                               \
  k1 = lop3<threshold_lut<NEED>(false, true, true)>(e01, e12, e13);                              \
  k2 = lop3<threshold_lut<NEED>(false, false, true)>(e02, e12, e23);                             \
  k3 = lop3<threshold_lut<NEED>(false, false, false)>(e03, e13, e23);                            \
}
    SDGP_KEEP4(rA0, rA1, rA2, rA3, a0, a1, a2, a3)
    SDGP_KEEP4(rB0, rB1, rB2, rB3, b0, b1, b2, b3)
#undef SDGP_KEEP4
    k.k0 = prmt(a0, b0, 0x7733); k.k1 = prmt(a1, b1, 0x7733);
    k.k2 = prmt(a2, b2, 0x7733); k.k3 = prmt(a3, b3, 0x7733);
  } else {
    // |x| as 15-bit integers, lanes (element i, element i + 4). d(i,j) = (a_i | 0x8000) - a_j per lane never borrows across
    // lanes and has bit 15 of the lane set iff a_i >= a_j, i.e. iff i beats j (i < j: ties to i).
    constexpr uint32_t H = 0x80008000u;
    const uint32_t l0 = prmt(w.x, w.z, 0x5410) & ~H, l1 = prmt(w.x, w.z, 0x7632) & ~H;
    const uint32_t l2 = prmt(w.y, w.w, 0x5410) & ~H, l3 = prmt(w.y, w.w, 0x7632) & ~H;
    const uint32_t h0 = l0 + H, h1 = l1 + H, h2 = l2 + H;
    const uint32_t d01 = h0 - l1, d02 = h0 - l2, d03 = h0 - l3, d12 = h1 - l2, d13 = h1 - l3,
                   d23 = h2 - l3;
    k.k0 = lop3<threshold_lut<NEED>(false, false, false)>(d01, d02, d03);
    k.k1 = lop3<threshold_lut<NEED>(true, false, false)>(d01, d12, d13);
    k.k2 = lop3<threshold_lut<NEED>(true, true, false)>(d02, d12, d23);
    k.k3 = lop3<threshold_lut<NEED>(true, true, true)>(d03, d13, d23);
  }
  return k;
}

// Gathers the slots of a vector: out.x / out.y = slots 0 and 1 (low and high half-word) of chunk A / B, pads +0.
// EXACT2: every chunk keeps exactly two elements (2:4), so there are no pads.
template <bool EXACT2>
__device__ __forceinline__ void gather_slots(const uint4& w, const KeepFlags& k, uint2& out, uint2& slot_mask, uint32_t& pos_top) {
  const uint32_t not0 = EXACT2 ? ~k.k0 : majority(k.k1, k.k2, k.k3);
  const uint32_t sel = chunk_selectors(not0, k);
  pos_top = positions_top_byte(sel);
  out = make_uint2(prmt(w.x, w.y, sel), prmt(w.z, w.w, sel >> 16));
  if (EXACT2) {
    slot_mask = make_uint2(0xFFFFFFFFu, 0xFFFFFFFFu);
  } else {
    // slot 0 holds a survivor if element 0 is kept or two are, slot 1 if anything but element 0 is
    const uint32_t keep0 = k.k0 | not0, keep1 = lop3<0xFE>(k.k1, k.k2, k.k3);
    slot_mask = make_uint2(prmt(keep0, keep1, 0xDD99), prmt(keep0, keep1, 0xFFBB));
    out.x &= slot_mask.x;
    out.y &= slot_mask.y;
  }
}

// The L1 rescale of Section 3.2 on gathered slots: `lo`, `hi` of a chunk's word times its group's scale, rounded to the
// element type. finite: both sums of the group are finite, so every product is (the hardware's packed rounding applies, and a
// +0 pad stays +0); otherwise each value goes through the explicit rounding (NaN stored as the canonical quiet NaN) and pads
// are masked (their product with a scale that is not finite is not +0).
template <bool F16>
__device__ __forceinline__ uint32_t rescale_slots(uint32_t word, float scale, bool finite, uint32_t mask) {
  const float lo = __fmul_rn(lane_lo<F16>(word), scale), hi = __fmul_rn(lane_hi<F16>(word), scale);
  if (finite) return pack_pair_rn<F16>(lo, hi);
  return (f32_to_elem_bits<F16>(lo) | (f32_to_elem_bits<F16>(hi) << 16)) & mask;
}

__device__ __forceinline__ bool is_finite(float x) { return (__float_as_uint(x) & 0x7F800000u) != 0x7F800000u; }

// Sum of the magnitudes of a word's two elements.
template <bool F16>
__device__ __forceinline__ float pair_abs(uint32_t word) { return __fadd_rn(lane_lo_abs<F16>(word), lane_hi_abs<F16>(word)); }

// m = 4: both groups of vector w (number v in the tensor) in compressed form. The rescaled function's sums are the oracle's
// (balanced pairwise in index order; over the survivors only the slots' terms are not +0, so that sum is one addition).
template <int N, int SCHEME, bool F16>
__device__ __forceinline__ void m4_compress(const uint4& w, int64_t v, uint32_t seed_lo, uint32_t seed_hi, uint2& out,
                                            uint32_t& pos_top, KeepFlags& k) {
  static_assert(N == 1 || N == 2, "a compressed form exists for one or two survivors");
  k = m4_flags<N, SCHEME == SDGP_RANDOM ? SDGP_RANDOM : SDGP_MAGNITUDE>(w, v, seed_lo, seed_hi);
  uint2 mask;
  gather_slots<N == 2>(w, k, out, mask, pos_top);
  if (SCHEME == SDGP_RESCALED_MAGNITUDE) {
    const float tA = __fadd_rn(pair_abs<F16>(w.x), pair_abs<F16>(w.y)), tB = __fadd_rn(pair_abs<F16>(w.z), pair_abs<F16>(w.w));
    const float sA = pair_abs<F16>(out.x), sB = pair_abs<F16>(out.y);
    const float scA = (sA == 0.0f) ? 1.0f : __fdiv_rn(tA, sA), scB = (sB == 0.0f) ? 1.0f : __fdiv_rn(tB, sB);
    const bool finite = is_finite(tA) && is_finite(tB);
    out.x = rescale_slots<F16>(out.x, scA, finite, mask.x);
    out.y = rescale_slots<F16>(out.y, scB, finite, mask.y);
  }
}

// Groups of 8, 16 or 32 with n <= 2 (Algorithm 1 with the same three pruning functions): the survivors are the
// elements whose composite key (rank key, then 31 - position: unique inside a group) reaches the group's n-th
// largest. The M / 8 vectors of a group are held by M / 8 neighbouring lanes (lane bits 0 and up; `part` = this
// lane's number among them, i.e. which eighth of the group the vector is); each lane finds the two largest keys
// of its 8 elements with a max/min network and the lanes merge their pairs through xor-shuffles, which every
// lane named in `lanes` must execute together. Output in the lane-paired form of m4_prune_vector.
__device__ __forceinline__ void merge_top2(uint32_t& hi, uint32_t& lo, uint32_t hi2, uint32_t lo2) {
  const uint32_t h = max(hi, hi2);
  lo = __vimax3_u32(min(hi, hi2), lo, lo2);
  hi = h;
}

// Composite keys (31 bits) of the 8 elements of vector w (number v in the tensor); pos0 = tie-break bits of element 0 (below
// 2^15). Magnitude: |x| in bits 16..30, so that an element in a word's upper half costs one logic operation and one in the
// lower half a shift more. Random: the complement of the 16-bit key in bits 15..30 (the smallest key ranks first).
// src: the vector itself, or (random function) its four words of random bits.
template <int SCHEME>
__device__ __forceinline__ void top2_keys_of(const uint4& src, uint32_t pos0, uint32_t (&c)[8]) {
  const uint32_t ww[4] = {src.x, src.y, src.z, src.w};
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    if (SCHEME == SDGP_RANDOM) c[i] = (~((i & 1) ? (ww[i >> 1] >> 1) : (ww[i >> 1] << 15)) & 0x7FFF8000u) | (pos0 - i);
    else c[i] = (((i & 1) ? ww[i >> 1] : (ww[i >> 1] << 16)) & 0x7FFF0000u) | (pos0 - i);
  }
}
template <int SCHEME>
__device__ __forceinline__ void top2_keys(const uint4& w, int64_t v, uint32_t seed_lo, uint32_t seed_hi, uint32_t pos0,
                                          uint32_t (&c)[8]) {
  if (SCHEME == SDGP_RANDOM)
    top2_keys_of<SCHEME>(philox4x32_10((uint32_t)v, (uint32_t)((uint64_t)v >> 32), 0u, 0u, seed_lo, seed_hi), pos0, c);
  else
    top2_keys_of<SCHEME>(w, pos0, c);
}

// The two largest of eight keys.
__device__ __forceinline__ void top2_of_8(const uint32_t (&c)[8], uint32_t& hi, uint32_t& lo) {
  uint32_t h1 = max(c[2], c[3]), l1 = min(c[2], c[3]), h2 = max(c[4], c[5]), l2 = min(c[4], c[5]),
           h3 = max(c[6], c[7]), l3 = min(c[6], c[7]);
  hi = max(c[0], c[1]);
  lo = min(c[0], c[1]);
  merge_top2(hi, lo, h1, l1);
  merge_top2(h2, l2, h3, l3);
  merge_top2(hi, lo, h2, l2);
}

// Lane-paired values and keep masks of a vector whose elements with key > t1 survive.
__device__ __forceinline__ void top2_apply(const uint4& w, const uint32_t (&c)[8], uint32_t t1, uint32_t& p0, uint32_t& p1,
                                           uint32_t& p2, uint32_t& p3, uint32_t& y0, uint32_t& y1, uint32_t& y2, uint32_t& y3,
                                           uint32_t& km0, uint32_t& km1, uint32_t& km2, uint32_t& km3) {
  p0 = prmt(w.x, w.z, 0x5410); p1 = prmt(w.x, w.z, 0x7632);
  p2 = prmt(w.y, w.w, 0x5410); p3 = prmt(w.y, w.w, 0x7632);
  km0 = prmt(t1 - c[0], t1 - c[4], 0xFFBB); km1 = prmt(t1 - c[1], t1 - c[5], 0xFFBB);  // (t1 - key) negative <=> kept
  km2 = prmt(t1 - c[2], t1 - c[6], 0xFFBB); km3 = prmt(t1 - c[3], t1 - c[7], 0xFFBB);
  y0 = p0 & km0; y1 = p1 & km1; y2 = p2 & km2; y3 = p3 & km3;
}

template <int M, int SCHEME, bool F16 = false>
__device__ __forceinline__ void top2_prune_vector(const uint4& w, int64_t v, uint32_t seed_lo, uint32_t seed_hi, int n,
                                                  int part, unsigned lanes, uint32_t& y0, uint32_t& y1, uint32_t& y2,
                                                  uint32_t& y3, uint32_t& km0, uint32_t& km1, uint32_t& km2,
                                                  uint32_t& km3) {
  constexpr int LANES = M / 8;
  uint32_t c[8], hi, lo;
  top2_keys<SCHEME>(w, v, seed_lo, seed_hi, 31u - 8u * (uint32_t)part, c);
  top2_of_8(c, hi, lo);
#pragma unroll
  for (int d = 1; d < LANES; d <<= 1) {
    const uint32_t oh = __shfl_xor_sync(lanes, hi, d), ol = __shfl_xor_sync(lanes, lo, d);
    merge_top2(hi, lo, oh, ol);
  }
  uint32_t p0, p1, p2, p3;
  top2_apply(w, c, ((n == 1) ? hi : lo) - 1u, p0, p1, p2, p3, y0, y1, y2, y3, km0, km1, km2, km3);
  if (SCHEME == SDGP_RESCALED_MAGNITUDE) {
    // balanced pairwise sums in index order: elements 0..3 are the low lanes, 4..7 the high lanes
    float tsum = __fadd_rn(sum4_lo_abs<F16>(p0, p1, p2, p3), sum4_hi_abs<F16>(p0, p1, p2, p3));
    float ssum = __fadd_rn(sum4_lo_abs<F16>(y0, y1, y2, y3), sum4_hi_abs<F16>(y0, y1, y2, y3));
#pragma unroll
    for (int d = 1; d < LANES; d <<= 1) {
      tsum = __fadd_rn(tsum, __shfl_xor_sync(lanes, tsum, d));
      ssum = __fadd_rn(ssum, __shfl_xor_sync(lanes, ssum, d));
    }
    const float sc = (ssum == 0.0f) ? 1.0f : __fdiv_rn(tsum, ssum);
    rescale_packed<F16>(y0, y1, y2, y3, km0, km1, km2, km3, sc, sc, tsum, tsum);
  }
}

// Keep flags in lane form of a vector whose elements with key > t1 survive.
__device__ __forceinline__ KeepFlags top2_flags(const uint32_t (&c)[8], uint32_t t1) {
  KeepFlags k;  // (t1 - key) negative <=> kept; the sign bits of elements i and i + 4 side by side
  k.k0 = prmt(t1 - c[0], t1 - c[4], 0x7733); k.k1 = prmt(t1 - c[1], t1 - c[5], 0x7733);
  k.k2 = prmt(t1 - c[2], t1 - c[6], 0x7733); k.k3 = prmt(t1 - c[3], t1 - c[7], 0x7733);
  return k;
}

// Groups of M = 8, 16 or 32 in compressed form (arguments as top2_prune_vector). A group keeps at most two elements, so in
// the rescaled function's sum over the survivors every term but the slots' is +0.
template <int M, int SCHEME, bool F16>
__device__ __forceinline__ void top2_compress(const uint4& w, int64_t v, uint32_t seed_lo, uint32_t seed_hi, int n, int part,
                                              unsigned lanes, uint2& out, uint32_t& pos_top, KeepFlags& k) {
  constexpr int LANES = M / 8;
  uint32_t c[8], hi, lo;
  top2_keys<SCHEME>(w, v, seed_lo, seed_hi, 31u - 8u * (uint32_t)part, c);
  top2_of_8(c, hi, lo);
#pragma unroll
  for (int d = 1; d < LANES; d <<= 1) {
    const uint32_t oh = __shfl_xor_sync(lanes, hi, d), ol = __shfl_xor_sync(lanes, lo, d);
    merge_top2(hi, lo, oh, ol);
  }
  k = top2_flags(c, ((n == 1) ? hi : lo) - 1u);
  uint2 mask;
  gather_slots<false>(w, k, out, mask, pos_top);
  if (SCHEME == SDGP_RESCALED_MAGNITUDE) {
    float tsum = __fadd_rn(__fadd_rn(pair_abs<F16>(w.x), pair_abs<F16>(w.y)), __fadd_rn(pair_abs<F16>(w.z), pair_abs<F16>(w.w)));
    float ssum = __fadd_rn(pair_abs<F16>(out.x), pair_abs<F16>(out.y));
#pragma unroll
    for (int d = 1; d < LANES; d <<= 1) {
      tsum = __fadd_rn(tsum, __shfl_xor_sync(lanes, tsum, d));
      ssum = __fadd_rn(ssum, __shfl_xor_sync(lanes, ssum, d));
    }
    const float sc = (ssum == 0.0f) ? 1.0f : __fdiv_rn(tsum, ssum);
    const bool finite = is_finite(tsum);
    out.x = rescale_slots<F16>(out.x, sc, finite, mask.x);
    out.y = rescale_slots<F16>(out.y, sc, finite, mask.y);
  }
}

// One vector of a group of M (4, 8, 16, 32) in compressed form: out and pos_top as gather_slots.
template <int M, int N, int SCHEME, bool F16>
__device__ __forceinline__ void compress_vector(const uint4& w, int64_t v, uint32_t seed_lo, uint32_t seed_hi, int part,
                                                unsigned lanes, uint2& out, uint32_t& pos_top, KeepFlags& k) {
  if constexpr (M == 4) m4_compress<N, SCHEME, F16>(w, v, seed_lo, seed_hi, out, pos_top, k);
  else top2_compress<M, SCHEME, F16>(w, v, seed_lo, seed_hi, N, part, lanes, out, pos_top, k);
}

// Two neighbouring vectors (numbers v and v + 1, v even) held by the same thread, in compressed form: both groups of an M = 8
// pair, the group of 16 they form, or half a group of 32 whose other half the lane with bit 0 flipped holds (`part` =
// which half this lane has; every lane named in `lanes` must call together).
template <int M, int N, int SCHEME, bool F16>
__device__ __forceinline__ void compress_pair(const uint4& wa, const uint4& wb, int64_t v, uint32_t seed_lo, uint32_t seed_hi,
                                              int part, unsigned lanes, uint4& out, uint32_t& posa, uint32_t& posb,
                                              KeepFlags& ka, KeepFlags& kb) {
  uint2 oa, ob;
  if constexpr (M <= 8) {
    compress_vector<M, N, SCHEME, F16>(wa, v, seed_lo, seed_hi, 0, lanes, oa, posa, ka);
    compress_vector<M, N, SCHEME, F16>(wb, v + 1, seed_lo, seed_hi, 0, lanes, ob, posb, kb);
  } else {
    uint32_t ca[8], cb[8], hi, lo, hb, lb;
    const uint32_t pos0 = 31u - 16u * (uint32_t)part;
    top2_keys<SCHEME>(wa, v, seed_lo, seed_hi, pos0, ca);
    top2_keys<SCHEME>(wb, v + 1, seed_lo, seed_hi, pos0 - 8u, cb);
    top2_of_8(ca, hi, lo);
    top2_of_8(cb, hb, lb);
    merge_top2(hi, lo, hb, lb);
    if (M == 32) merge_top2(hi, lo, __shfl_xor_sync(lanes, hi, 1), __shfl_xor_sync(lanes, lo, 1));
    const uint32_t t1 = ((N == 1) ? hi : lo) - 1u;
    ka = top2_flags(ca, t1);
    kb = top2_flags(cb, t1);
    uint2 ma, mb;
    gather_slots<false>(wa, ka, oa, ma, posa);
    gather_slots<false>(wb, kb, ob, mb, posb);
    if (SCHEME == SDGP_RESCALED_MAGNITUDE) {
      // the oracle's tree: (elements 0..7) + (elements 8..15), then the other sixteen
      float tsum = __fadd_rn(__fadd_rn(__fadd_rn(pair_abs<F16>(wa.x), pair_abs<F16>(wa.y)), __fadd_rn(pair_abs<F16>(wa.z), pair_abs<F16>(wa.w))),
                             __fadd_rn(__fadd_rn(pair_abs<F16>(wb.x), pair_abs<F16>(wb.y)), __fadd_rn(pair_abs<F16>(wb.z), pair_abs<F16>(wb.w))));
      float ssum = __fadd_rn(__fadd_rn(pair_abs<F16>(oa.x), pair_abs<F16>(oa.y)), __fadd_rn(pair_abs<F16>(ob.x), pair_abs<F16>(ob.y)));
      if (M == 32) {
        tsum = __fadd_rn(tsum, __shfl_xor_sync(lanes, tsum, 1));
        ssum = __fadd_rn(ssum, __shfl_xor_sync(lanes, ssum, 1));
      }
      const float sc = (ssum == 0.0f) ? 1.0f : __fdiv_rn(tsum, ssum);
      const bool finite = is_finite(tsum);
      oa = make_uint2(rescale_slots<F16>(oa.x, sc, finite, ma.x), rescale_slots<F16>(oa.y, sc, finite, ma.y));
      ob = make_uint2(rescale_slots<F16>(ob.x, sc, finite, mb.x), rescale_slots<F16>(ob.y, sc, finite, mb.y));
    }
  }
  out = make_uint4(oa.x, oa.y, ob.x, ob.y);
}

// One group of 32 whose four vectors (numbers v .. v + 3) are held by the same thread, in compressed form. The keys are made
// twice, once for the two largest and once for the decision: 32 of them at a time do not fit the registers.
template <int N, int SCHEME, bool F16>
__device__ __forceinline__ void compress_quad32(const uint4 (&w)[4], int64_t v, uint32_t seed_lo, uint32_t seed_hi, uint2 (&out)[4],
                                                uint32_t (&pos)[4]) {
  uint4 r[4];  // random function: the keys' source, generated once
  uint32_t hi = 0u, lo = 0u;
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    if (SCHEME == SDGP_RANDOM) r[t] = philox4x32_10((uint32_t)(v + t), (uint32_t)((uint64_t)(v + t) >> 32), 0u, 0u, seed_lo, seed_hi);
    uint32_t c[8], h, l;
    top2_keys_of<SCHEME>(SCHEME == SDGP_RANDOM ? r[t] : w[t], 31u - 8u * t, c);
    top2_of_8(c, h, l);
    if (t == 0) { hi = h; lo = l; }
    else merge_top2(hi, lo, h, l);
  }
  const uint32_t t1 = ((N == 1) ? hi : lo) - 1u;
  uint2 mask[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    uint32_t c[8];
    top2_keys_of<SCHEME>(SCHEME == SDGP_RANDOM ? r[t] : w[t], 31u - 8u * t, c);
    gather_slots<false>(w[t], top2_flags(c, t1), out[t], mask[t], pos[t]);
  }
  if (SCHEME == SDGP_RESCALED_MAGNITUDE) {
    float ts[4], ss[4];  // the oracle's tree, eight elements at a time
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      ts[t] = __fadd_rn(__fadd_rn(pair_abs<F16>(w[t].x), pair_abs<F16>(w[t].y)), __fadd_rn(pair_abs<F16>(w[t].z), pair_abs<F16>(w[t].w)));
      ss[t] = __fadd_rn(pair_abs<F16>(out[t].x), pair_abs<F16>(out[t].y));
    }
    const float tsum = __fadd_rn(__fadd_rn(ts[0], ts[1]), __fadd_rn(ts[2], ts[3]));
    const float ssum = __fadd_rn(__fadd_rn(ss[0], ss[1]), __fadd_rn(ss[2], ss[3]));
    const float sc = (ssum == 0.0f) ? 1.0f : __fdiv_rn(tsum, ssum);
    const bool finite = is_finite(tsum);
#pragma unroll
    for (int t = 0; t < 4; ++t)
      out[t] = make_uint2(rescale_slots<F16>(out[t].x, sc, finite, mask[t].x), rescale_slots<F16>(out[t].y, sc, finite, mask[t].y));
  }
}

}  // namespace
}  // namespace sdgp
