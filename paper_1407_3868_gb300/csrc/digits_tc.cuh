// Products of 48-bit fixed-point operands on the tensor cores, shared by the FP64 translation
// (translate_f64_tc.cu) and the FP64 contour contractions (contour_f64_tc.cu).
//
// Both operands W (128 rows per CTA) and X (NPAD columns) are cut into six balanced 8-bit digits held
// as FP16 integers; digit products have at most 14 bits and the FP32 accumulators sum them exactly
// while a level's sum stays below 2^24: levels 0 to 3 collect at most four products per K value, so
// 256 K values always fit before the accumulators are drained into 64-bit integers.  The lowest levels
// may leave the exact range; their unit is far below what is left out.  Level L collects the products of W digit i and X digit j with
// i + j = L, weight 2^(8 (10 - L)); its NPAD columns follow those of level L - 1 in tensor memory, so
// that one tcgen05.mma of W plane i with several X planes side by side in N fills consecutive levels.
//
// Shared memory of a stage, K-major core matrices of 8 rows x 16 bytes without swizzle: six W planes
// [K group][row][8 K values], then X [K group][plane][column][8 K values].  A thread that owns a row
// writes 16 bytes next to its neighbour's, and X is copied as it lies in global memory.
#pragma once

#include <cuda_fp16.h>

#include "fixed64.cuh"
#include "tc_ptx.cuh"

namespace {

constexpr int PL = 6;                         // digit planes of either operand
constexpr int ROWS = 128;                     // rows of W (MMA M) per CTA
constexpr int KG = 4;                         // groups of 8 K values per stage: two MMA steps of K = 16
constexpr int A_KG = ROWS * 16;               // bytes of one K group of one plane
constexpr int A_PLANE = KG * A_KG;
constexpr int A_BYTES = PL * A_PLANE;         // 49152
constexpr int STAGES = 3;
constexpr int DRAIN_WARPS = 8;
constexpr int DRAIN = 8;                      // stages per drain: 256 K values, 4 products x 256 x 2^14 = 2^24

__host__ __device__ constexpr int b_kg_bytes(int npad) { return PL * npad * 16; }
__host__ __device__ constexpr int stage_bytes(int npad) { return A_BYTES + KG * b_kg_bytes(npad); }
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

// The six balanced digits of two 48-bit values (bits 16..63 of wa and wb less kDigitBias, most
// significant first) as pairs of FP16 integers in [-128, 127]: byte + 128 sits in the low mantissa
// bits of 1024 + byte.
constexpr uint64_t kDigitBias = 0x8080808080808000ull;   // +128 per digit, and half a unit to round
__device__ __forceinline__ void biased_digit_pairs(uint64_t wa, uint64_t wb, uint32_t* out) {
  const uint32_t ah = (uint32_t)(wa >> 32), al = (uint32_t)wa, bh = (uint32_t)(wb >> 32), bl = (uint32_t)wb;
  const uint32_t t0 = __byte_perm(ah, bh, 0x6273);  // a3 b3 a2 b2 (byte 3 the most significant)
  const uint32_t t1 = __byte_perm(ah, bh, 0x4051);  // a1 b1 a0 b0
  const uint32_t t2 = __byte_perm(al, bl, 0x6273);  // the two top bytes of the low words
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
}
__device__ __forceinline__ void digit_pairs(int64_t a, int64_t b, uint32_t* out) {
  biased_digit_pairs((uint64_t)a + kDigitBias, (uint64_t)b + kDigitBias, out);
}

// Levels of one accumulated element -> units of level 5 / 64, added to acc.
template <int LMAX>
__device__ __forceinline__ void add_levels(int64_t& acc, const uint32_t* f) {
  int lo = __float2int_rn(__uint_as_float(f[5]));
  if (LMAX >= 6) lo += (__float2int_rn(__uint_as_float(f[6])) + 128) >> 8;
  acc = mad_wide((lo + 32) >> 6, 1, acc);
  acc = mad_wide(__float2int_rn(__uint_as_float(f[4])), 1 << 2, acc);
  acc = mad_wide(__float2int_rn(__uint_as_float(f[3])), 1 << 10, acc);
  acc = mad_wide(__float2int_rn(__uint_as_float(f[2])), 1 << 18, acc);
  acc = mad_wide(__float2int_rn(__uint_as_float(f[1])), 1 << 26, acc);
  acc = mad_wide(__float2int_rn(__uint_as_float(f[0])) * 16, 1 << 30, acc);
}

constexpr unsigned long long kInfBits = 0x7ff0000000000000ull;
// e with the value <= 0.99 2^e (bits of a non-negative double): 48-bit balanced digits in units of
// 2^(e - 47) hold it, in units of 2^(e - 46) the sum of two
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

// The MMAs of step `ks` of the stage at sa (W) and sb (X); `first`: the step that starts
// the accumulators (W plane 0 covers levels 0..5; level 6 starts with W plane 1 and X plane 5, issued
// apart).
template <int NPAD, int LMAX>
__device__ __forceinline__ void issue_step(uint32_t tmem, uint32_t sa, uint32_t sb, int ks, bool first) {
  constexpr int MAXPL = 256 / NPAD;              // planes of X one MMA takes
  constexpr uint32_t B_KG = b_kg_bytes(NPAD);
#pragma unroll
  for (int i = 0; i < PL; ++i) {
    const uint64_t da = core_desc(sa + i * A_PLANE + ks * 2 * A_KG, A_KG);
    const int jn = LMAX + 1 - i < PL ? LMAX + 1 - i : PL;
#pragma unroll
    for (int j0 = 0; j0 < PL; j0 += MAXPL) {
      if (j0 >= jn) continue;
      int jc = jn - j0 < MAXPL ? jn - j0 : MAXPL;
      const bool split6 = first && LMAX >= 6 && i == 1 && j0 + jc == PL;
      if (split6) --jc;
      if (jc > 0)
        mma_bf16(tmem + (i + j0) * NPAD, da, core_desc(sb + ks * 2 * B_KG + j0 * NPAD * 16, B_KG),
                 idesc_f16(ROWS, jc * NPAD), !(first && i == 0));
      if (split6)
        mma_bf16(tmem + 6 * NPAD, da, core_desc(sb + ks * 2 * B_KG + 5 * NPAD * 16, B_KG), idesc_f16(ROWS, NPAD), 0);
    }
  }
}

// Add the accumulators of this warp's 32 rows and NPAD / 2 columns (tb: its tensor-memory address) to
// acc, in units of 2^46 = 64 of level 5.
template <int NPAD, int LMAX>
__device__ __forceinline__ void drain_levels(uint32_t tb, int64_t* acc) {
  constexpr int NL = LMAX + 1;
#pragma unroll
  for (int cb = 0; cb < NPAD / 8; ++cb) {
    uint32_t f[NL][4];
#pragma unroll
    for (int L = 0; L < NL; ++L) tmem_ld4(tb + L * NPAD + 4 * cb, f[L]);
    tmem_wait_ld();
#pragma unroll
    for (int L = 0; L < NL; ++L)               // keep every use of the loaded registers behind the wait
      asm volatile("" : "+r"(f[L][0]), "+r"(f[L][1]), "+r"(f[L][2]), "+r"(f[L][3]));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      uint32_t e[NL];
#pragma unroll
      for (int L = 0; L < NL; ++L) e[L] = f[L][i];
      add_levels<LMAX>(acc[4 * cb + i], e);
    }
  }
}

}  // namespace
