// Products of fixed-point operands on the tensor cores, shared by the FP64 translation
// (translate_f64_tc.cu: 48-bit operands, six digits) and the FP64 contour contractions
// (contour_f64_tc.cu: 56-bit operands, seven digits).
//
// Both operands W (128 rows per CTA) and X (NPAD columns) are cut into balanced 8-bit digits held as
// FP16 integers; digit products have at most 14 bits and the FP32 accumulators sum them exactly while
// a level's sum stays below 2^24.  Level L collects the products of W digit i and X digit j with
// i + j = L, at most L + 1 of them per K value: level L is exact over 1024 / (L + 1) K values whatever
// the digits; beyond that its sums may be rounded to their 24 leading bits.  The accumulators are
// drained into 64-bit integers.  The NPAD columns of level L follow those of level L - 1 in tensor
// memory, so that one tcgen05.mma of W plane i with several X planes side by side in N fills
// consecutive levels.
//
// Shared memory of a stage, K-major core matrices of 8 rows x 16 bytes without swizzle: the W planes
// [K group][row][8 K values], then X [K group][plane][column][8 K values].  A thread that owns a row
// writes 16 bytes next to its neighbour's, and X is copied as it lies in global memory.
#pragma once

#include <cuda_fp16.h>

#include "fixed64.cuh"
#include "tc_ptx.cuh"

namespace {

constexpr int ROWS = 128;                     // rows of W (MMA M) per CTA
constexpr int A_KG = ROWS * 16;               // bytes of one K group (8 K values) of one plane
constexpr int DRAIN_WARPS = 8;

// `planes` digits of either operand, stages of `groups` K groups (two make an MMA step of K = 16)
template <int PLANES, int GROUPS_>
struct DigitTile {
  static constexpr int PL = PLANES, KG = GROUPS_;
  static constexpr int A_PLANE = KG * A_KG;
  static constexpr int A_BYTES = PL * A_PLANE;
  static __host__ __device__ constexpr int b_kg_bytes(int npad) { return PL * npad * 16; }
  static __host__ __device__ constexpr int stage_bytes(int npad) { return A_BYTES + KG * b_kg_bytes(npad); }
};
// columns of one digit plane of X: Re and Im of 2p + 1 orders, padded to the MMA's granularity
// (16 columns for any number of planes side by side)
inline int pad_columns(int p) { return p <= 7 ? 32 : p <= 11 ? 48 : 64; }

// Instruction descriptor, kind::f16: D = F32, A = B = F16, both K-major, M x N.
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// Shared-memory descriptor, K-major without swizzle: core matrices of 8 rows x 16 bytes (128 bytes,
// contiguous); `lead` bytes to the next core matrix along K, 128 bytes to the next 8 rows.
__device__ __forceinline__ uint64_t core_desc(uint32_t saddr, uint32_t lead) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | (uint64_t)(lead >> 4) << 16 | (uint64_t)(128 >> 4) << 32 |
         (uint64_t)1 << 46;
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t* v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// The N balanced digits of two 64-bit values (their N top bytes, rounded; the values come with
// digit_bias<N> added; most significant first) as pairs of FP16 integers in [-128, 127]: byte + 128 sits
// in the low mantissa bits of 1024 + byte.
template <int N>
__host__ __device__ constexpr uint64_t digit_bias() {   // +128 per digit, and half a unit to round
  return N == 6 ? 0x8080808080808000ull : 0x8080808080808080ull;
}
template <int N>
__device__ __forceinline__ void biased_digit_pairs(uint64_t wa, uint64_t wb, uint32_t* out) {
  static_assert(N == 6 || N == 7, "digits");
  const uint32_t ah = (uint32_t)(wa >> 32), al = (uint32_t)wa, bh = (uint32_t)(wb >> 32), bl = (uint32_t)wb;
  const uint32_t t0 = __byte_perm(ah, bh, 0x6273);  // a3 b3 a2 b2 (byte 3 the most significant)
  const uint32_t t1 = __byte_perm(ah, bh, 0x4051);  // a1 b1 a0 b0
  const uint32_t t2 = __byte_perm(al, bl, 0x6273);  // the same of the low words
  const __half2 off = __float2half2_rn(1152.0f);
  const uint32_t one = 0x64646464u;
  auto pair = [&](uint32_t t, uint32_t sel) {
    const uint32_t w = __byte_perm(t, one, sel);
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w), off);
    return *reinterpret_cast<const uint32_t*>(&h);
  };
  out[0] = pair(t0, 0x4140);
  out[1] = pair(t0, 0x4342);
  out[2] = pair(t1, 0x4140);
  out[3] = pair(t1, 0x4342);
  out[4] = pair(t2, 0x4140);
  out[5] = pair(t2, 0x4342);
  if (N == 7) out[6] = pair(__byte_perm(al, bl, 0x4051), 0x4140);
}
template <int N>
__device__ __forceinline__ void digit_pairs(int64_t a, int64_t b, uint32_t* out) {
  biased_digit_pairs<N>((uint64_t)a + digit_bias<N>(), (uint64_t)b + digit_bias<N>(), out);
}

constexpr unsigned long long kInfBits = 0x7ff0000000000000ull;
// e with the value <= 0.99 2^e (bits of a non-negative double): N balanced digits in units of
// 2^(e - 8 N + 1) hold it, in units of 2^(e - 8 N + 2) the sum of two
__device__ __forceinline__ int scale_exponent(unsigned long long bits) {
  int e;
  const double m = frexp(__longlong_as_double((long long)bits), &e);
  return m > 0.99 ? e + 1 : e;
}

// v 2^ex, rounded to nearest, in integer instructions (the FP64 pipe takes 64 cycles of a scheduler
// per warp instruction).
__device__ __forceinline__ double fixed_to_double(int64_t v, int ex) {
  if (v == 0) return 0.0;
  const uint64_t u = v < 0 ? 0ull - (uint64_t)v : (uint64_t)v;
  const int lz = __clzll((long long)u);
  const uint64_t m = u << lz;
  const uint64_t keep = (m >> 11) + ((m >> 10) & 1);          // 53 bits, or 2^53
  const int e = 63 - lz + ex + 1022;                          // exponent field less one: keep brings the other
  if (e < 1 || e > 2044) return scalbn(scalbn(__ll2double_rn(v), ex / 2), ex - ex / 2);
  const uint64_t bits = ((uint64_t)e << 52) + keep;
  return __longlong_as_double((long long)(v < 0 ? bits | 0x8000000000000000ull : bits));
}

// The MMAs of step `ks` of the stage at sa (W) and sb (X), levels 0..LMAX; `first`: the step that starts
// the accumulators (W plane 0 covers the levels 0..PL - 1; a further one starts with W plane 1 and the
// last X plane, issued apart).
template <class Tile, int NPAD, int LMAX>
__device__ __forceinline__ void issue_step(uint32_t tmem, uint32_t sa, uint32_t sb, int ks, bool first) {
  constexpr int PL = Tile::PL, MAXPL = 256 / NPAD;   // planes of X one MMA takes
  constexpr uint32_t B_KG = Tile::b_kg_bytes(NPAD);
  static_assert(LMAX <= PL, "a level that starts with W plane 2");
#pragma unroll
  for (int i = 0; i < PL; ++i) {
    const uint64_t da = core_desc(sa + i * Tile::A_PLANE + ks * 2 * A_KG, A_KG);
    const int jn = LMAX + 1 - i < PL ? LMAX + 1 - i : PL;
#pragma unroll
    for (int j0 = 0; j0 < PL; j0 += MAXPL) {
      if (j0 >= jn) continue;
      int jc = jn - j0 < MAXPL ? jn - j0 : MAXPL;
      const bool split = first && LMAX >= PL && i == 1 && j0 + jc == PL;
      if (split) --jc;
      if (jc > 0)
        mma_bf16(tmem + (i + j0) * NPAD, da, core_desc(sb + ks * 2 * B_KG + j0 * NPAD * 16, B_KG),
                 idesc_f16(ROWS, jc * NPAD), !(first && i == 0));
      if (split)
        mma_bf16(tmem + PL * NPAD, da, core_desc(sb + ks * 2 * B_KG + (PL - 1) * NPAD * 16, B_KG),
                 idesc_f16(ROWS, NPAD), 0);
    }
  }
}

// Levels 0..LMAX of four columns of this warp's 32 rows from tensor memory (taddr: the first's level 0).
template <int NPAD, int LMAX>
__device__ __forceinline__ void load_levels(uint32_t taddr, uint32_t (*f)[4]) {
#pragma unroll
  for (int L = 0; L <= LMAX; ++L) tmem_ld4(taddr + L * NPAD, f[L]);
  tmem_wait_ld();
#pragma unroll
  for (int L = 0; L <= LMAX; ++L)              // keep every use of the loaded registers behind the wait
    asm volatile("" : "+r"(f[L][0]), "+r"(f[L][1]), "+r"(f[L][2]), "+r"(f[L][3]));
}

}  // namespace
