// FP64 translation of all pairs on the tensor cores (Sec. 3.2 Lemma 3.1), for one or more
// right-hand sides.
//
// The Toeplitz block of a pair holds h_s = H_s(k rho) e^{i s phi}, s = n - nu.  With A_s = J_s cos s phi,
// B_s = J_s sin s phi, C_s = Y_s cos s phi, D_s = Y_s sin s phi (s = 0..2p)
//   h_s = (A_s - D_s) + i (B_s + C_s),   h_{-s} = (-1)^s [(A_s + D_s) + i (C_s - B_s)],
// so the outputs of 128 targets are one real product summed over the sources,
//   alpha[target][(nu, Re/Im)] = sum_source sum_{s, A..D} W[target][(s, A..D)] X_source[(s, A..D)][(nu, Re/Im)],
// with X_source the signed sums beta_{nu+s} +- beta_{nu-s}.  W and X are held as 48-bit fixed point
// numbers (W: 48 fractional bits; X: relative to the largest coefficient of the
// right-hand side) and cut into six signed 8-bit digits each; the digits are exact in FP16, a product
// of two has at most 14 bits, so the tensor cores' FP32 sums are exact integers up to 2^24.  Products of
// digits i of W and j of X with i + j = L add into one accumulator per level L; levels beyond 5 or 6
// are below the 48 bits and left out (six_levels).  A row is as accurate as an FP64 sum's where the
// largest coefficient is a term of it, or one of its size is; k_dominant_row sums the only row that can be
// without.  One tcgen05.mma multiplies a digit plane of W with several
// digit planes of X side by side in N: its output columns are consecutive levels.
//
// Why: this chip's FP64 pipe (2 FMA per SM and clock) bounds the direct form at 133 ms for 5000 discs
// (k_translate_f64_sym: 168 ms); 21 products of FP16 digits take 4.7 ms at the tensor cores' measured
// rate, and this kernel 8.4 ms (1000 discs at p = 12, 26 products: 5.2 -> 0.33 ms).
//
// A CTA owns 128 targets and a range of sources.  Two warpgroups form the W rows of every second
// source each (thread = target; the fixed-point sequence of pair_fixed.cuh), eight orders at a time
// into the stage ring (consecutive threads write consecutive 16-byte pieces); warp 17 copies the X
// digits of the same orders (packed once per application); warp 16 issues the MMAs; warps 8-15 drain
// the accumulators into 64-bit integers, so a CTA's sum does not depend on any order.  When: before a
// round (two sources) whose X digits could carry a sum of the levels 0..4 past 2^24, from the bound
// that the packing kernel left for each source; the decaying coefficients of scattering problems let
// several rounds pass.  (One round alone stays below it in the levels 0..3 for any digits; in level 4
// only digits near +-128 nearly throughout could pass it, and be rounded to 2^-46 of the scales.)
// The ring holds three stages of two MMA steps: six stages of one step took 10.0 instead of 9.1 ms
// (5000 discs, the translation's part of the operator), a third warpgroup brought nothing.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "c64.cuh"
#include "digits_tc.cuh"
#include "lsms_internal.h"
#include "lsms_ops.h"
#include "near_f64.cuh"
#include "pair_fixed.cuh"

namespace {

using Tile = DigitTile<6, 4>;
constexpr int PL = Tile::PL, KG = Tile::KG, A_PLANE = Tile::A_PLANE, A_BYTES = Tile::A_BYTES, STAGES = 3;
__host__ __device__ constexpr int b_kg_bytes(int npad) { return Tile::b_kg_bytes(npad); }
__host__ __device__ constexpr int stage_bytes(int npad) { return Tile::stage_bytes(npad); }
constexpr int TABLE_BYTES = 256 * 16;
constexpr int kExact = 1 << 24;                // FP32 sums of integers are exact up to here
constexpr int MAX_SOURCES = 1024;             // per CTA: the 64-bit sums keep 10 bits for them
constexpr int GROUPS = 2;                     // warpgroups forming W
constexpr int GEN_WARPS = 4 * GROUPS;
constexpr int MMA_WARP = GEN_WARPS + DRAIN_WARPS;
constexpr int THREADS = (MMA_WARP + 2) * 32;
constexpr size_t smem_bytes(int npad) {
  return (size_t)STAGES * stage_bytes(npad) + TABLE_BYTES + MAX_SOURCES / GROUPS * sizeof(int) + 256;
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

// Add the accumulators of this warp's 32 rows and NPAD / 2 columns (tb: its tensor-memory address) to
// acc, in units of 2^46 = 64 of level 5.
template <int NPAD, int LMAX>
__device__ __forceinline__ void drain_levels(uint32_t tb, int64_t* acc) {
  constexpr int NL = LMAX + 1;
#pragma unroll
  for (int cb = 0; cb < NPAD / 8; ++cb) {
    uint32_t f[NL][4];
    load_levels<NPAD, LMAX>(tb + 4 * cb, f);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      uint32_t e[NL];
#pragma unroll
      for (int L = 0; L < NL; ++L) e[L] = f[L][i];
      add_levels<LMAX>(acc[4 * cb + i], e);
    }
  }
}

inline int k_steps(int p) { return (4 * (2 * p + 1) + 15) / 16; }   // K = 16 steps of one source

// What the digits of a right-hand side rest on: its largest |Re|, |Im| (the bits of a non-negative double;
// NaN and Inf compare above every finite value), the number of discs with a coefficient of at least
// 1/16 of it, and one such disc.
struct RhsStats {
  unsigned long long maxbits;
  int count, disc;
};

// Largest |Re|, |Im| of every disc (a warp each) and of each right-hand side.
__global__ void __launch_bounds__(256)
k_disc_max(const double2* __restrict__ x, int n, int P, unsigned long long* __restrict__ dmax,
           RhsStats* __restrict__ stats) {
  __shared__ unsigned long long part[8];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, r = blockIdx.y, l = blockIdx.x * 8 + w;
  unsigned long long m = 0;
  if (l < n && lane < P) {
    const double2 v = x[((size_t)r * n + l) * P + lane];
    m = max((unsigned long long)__double_as_longlong(v.x) & 0x7fffffffffffffffull,
            (unsigned long long)__double_as_longlong(v.y) & 0x7fffffffffffffffull);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) {
    part[w] = m;
    if (l < n) dmax[(size_t)r * n + l] = m;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < 8; ++i) m = max(m, part[i]);
    if (m) atomicMax(&stats[r].maxbits, m);
  }
}

// The large discs of each right-hand side, one CTA each (counted by the CTAs of k_pack_digits, whose updates
// of one address wait for each other, they took 14 us more at 2000 discs).
__global__ void __launch_bounds__(256)
k_large_discs(int n, const unsigned long long* __restrict__ dmax, RhsStats* __restrict__ stats) {
  __shared__ int part[8], disc;
  const int r = blockIdx.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned long long mb = stats[r].maxbits;
  const unsigned long long large = mb > (5ull << 52) ? mb - (4ull << 52) : 1;
  int count = 0;
  for (int l = threadIdx.x; l < n; l += 256)
    if (dmax[(size_t)r * n + l] >= large) {
      ++count;
      disc = l;
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) count += __shfl_xor_sync(0xffffffffu, count, o);
  if (lane == 0) part[w] = count;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < 8; ++i) count += part[i];
    stats[r].count = count;
    stats[r].disc = disc;
  }
}

// Digits of X for the sources src0 .. src0 + gridDim.x - 1 of right-hand side r0 + blockIdx.y:
// per source [K group][plane][column][8 K values] FP16, K = 4 s + (A, B, C, D), column 2 q + (Re, Im); and
// bound[source]: what the source adds to any element of the levels 0..4 at most, 128 sum |X digits of the
// planes 0..4|, or to a quarter of level 5, whose sums may pass 2^24 up to 2^26 (rounded to 2^-51
// of the scales).
__global__ void __launch_bounds__(256)
k_pack_digits(const double2* __restrict__ xs, int n, int p, int src0, int r0, int npad, int kgs,
              const RhsStats* __restrict__ stats, unsigned char* __restrict__ img, int* __restrict__ bound) {
  __shared__ long long re[128], im[128];          // beta_{nu +- s} at 48 + order, zero outside -p..p
  __shared__ int l1[64];                          // sum of |digit| per column, see the bound
  const int P = 2 * p + 1, r = r0 + blockIdx.y;
  const unsigned long long mb = stats[r].maxbits;
  if (mb == 0 || mb >= kInfBits) return;          // the product does not read the image then
  const int sh = 46 - scale_exponent(mb);
  const double2* b = xs + ((size_t)r * n + src0 + blockIdx.x) * P;
  if (threadIdx.x < 64) l1[threadIdx.x] = 0;
  if (threadIdx.x < 128) {
    const int o = (int)threadIdx.x - 48 + p;
    double2 v = make_double2(0.0, 0.0);
    if (o >= 0 && o < P) v = b[o];
    re[threadIdx.x] = llrint(scalbn(v.x, sh));
    im[threadIdx.x] = llrint(scalbn(v.y, sh));
  }
  __syncthreads();
  uint4* dst = (uint4*)(img + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * kgs * b_kg_bytes(npad));
  for (int it = threadIdx.x; it < kgs * npad; it += blockDim.x) {
    const int kg = it / npad, col = it - kg * npad;
    const int q = col >> 1, imag = col & 1;
    uint32_t w[PL][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int s = 2 * kg + h;
      long long a = 0, bb = 0, cc = 0, d = 0;
      if (q < P && s <= 2 * p) {
        const int c0 = 48 + q - p;
        const long long pr = re[c0 + s], pi = im[c0 + s];
        long long mr = 0, mi = 0;                 // (-1)^s beta_{nu - s}; s = 0 has one term only
        if (s > 0) {
          mr = re[c0 - s];
          mi = im[c0 - s];
          if (s & 1) { mr = -mr; mi = -mi; }
        }
        if (!imag) {
          a = pr + mr; bb = -pi + mi; cc = -pi - mi; d = -pr + mr;
        } else {
          a = pi + mi; bb = pr - mr; cc = pr + mr; d = -pi + mi;
        }
        if (s == 0) bb = d = 0;
        if (s & 2) { a = -a; bb = -bb; cc = -cc; d = -d; }   // the sequence's signs + + - -
      }
      uint32_t u[PL], v[PL];
      digit_pairs<PL>(a << 16, bb << 16, u);
      digit_pairs<PL>(cc << 16, d << 16, v);
#pragma unroll
      for (int j = 0; j < PL; ++j) {
        w[j][2 * h] = u[j];
        w[j][2 * h + 1] = v[j];
      }
    }
    int sum = 0, last = 0;
#pragma unroll
    for (int j = 0; j < PL; ++j) {
      dst[((size_t)kg * PL + j) * npad + col] = make_uint4(w[j][0], w[j][1], w[j][2], w[j][3]);
      __half2 h = __float2half2_rn(0.0f);         // four digits of at most 128 in a half: exact
#pragma unroll
      for (int i = 0; i < 4; ++i) h = __hadd2(h, __habs2(*reinterpret_cast<const __half2*>(&w[j][i])));
      const int d = (int)__low2float(h) + (int)__high2float(h);
      if (j < 5) sum += d;
      else last = d;
    }
    atomicAdd(&l1[col], max(sum, (sum + last + 3) / 4));
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    int m = max(l1[threadIdx.x], l1[threadIdx.x + 32]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (threadIdx.x == 0) bound[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = 128 * m;
  }
}

// Seven levels, or six: what six leave out is 1.3e-15 of the largest coefficient per term.  On right-hand
// sides whose discs are of one size (a quarter of them within 1/16 of the largest) the operator's
// translation is then 1.5e-12 off 64-bit sums at 1500 discs, 2.6e-13 with seven levels at 1000, 3.7e-12 and 4.2e-12 in
// the FP64 pipe's kernels; with one disc 1e4 larger six levels reach 1.4e-11.  Six spare 5 of 26 digit
// products, which counts where the products bound the kernel, from about 1024 discs on.
__device__ __forceinline__ bool six_levels(int n, int large_discs) { return n >= 1024 && large_discs >= n / 4; }

// grid: (target tiles, source ranges, right-hand sides); sources src0 + [0, nsrc) of the image; targets
// row0 .. row0 + nrows - 1, alpha holds those rows.  The row of a disc that is the only large one of its
// right-hand side is left to k_dominant_row.
template <int NPAD>
__global__ void __launch_bounds__(THREADS, 1)
k_translate_digits(const double* __restrict__ cx, const double* __restrict__ cy, int n, int p, PairConsts pc,
                   const longlong2* __restrict__ table, const unsigned char* __restrict__ img,
                   const int* __restrict__ bound, int src0, int nsrc,
                   int per_cta, int r0, const RhsStats* __restrict__ stats, int row0, int nrows,
                   double2* __restrict__ alpha, int* __restrict__ err) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int STAGE = stage_bytes(NPAD);
  longlong2* stab = (longlong2*)(smem + STAGES * STAGE);
  int* round_bound = (int*)(smem + STAGES * STAGE + TABLE_BYTES);      // [rounds]
  uint64_t* bars = (uint64_t*)(round_bound + MAX_SOURCES / GROUPS);   // full[S], empty[S], acc_full, acc_empty
  uint32_t* tmem_slot = (uint32_t*)(bars + 2 * STAGES + 2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int P = 2 * p + 1, r = r0 + blockIdx.z;
  const int s_begin = blockIdx.y * per_cta, s_end = min(nsrc, s_begin + per_cta);
  const RhsStats stat = stats[r];
  const unsigned long long mb = stat.maxbits;
  const bool six = six_levels(n, stat.count);
  double2* ar = alpha + (size_t)r * nrows * P;
  if (s_begin >= s_end || mb == 0) return;
  if (mb >= kInfBits) {                            // a non-finite coefficient reaches every target
    if (blockIdx.y == 0) {
      const double nan = __longlong_as_double(0x7ff8000000000000ll);
      for (int i = threadIdx.x; i < ROWS * P; i += THREADS) {
        const size_t e = (size_t)blockIdx.x * ROWS * P + i;
        if (e < (size_t)nrows * P) ar[e] = make_double2(nan, nan);
      }
    }
    return;
  }
  const int steps = (4 * P + 15) / 16;             // K = 16 steps of a source
  const int rounds = (s_end - s_begin + GROUPS - 1) / GROUPS;
  const int chunks = (steps + 1) / 2;              // stages of a source
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * STAGES, accf = full0 + 16 * STAGES, acce = accf + 8;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full0 + 8 * s, 5);                 // four forming warps and the copy
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(accf, 1);
    mbar_init(acce, DRAIN_WARPS);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x < 256) stab[threadIdx.x] = table[threadIdx.x];
  for (int q = threadIdx.x; q < rounds; q += THREADS) {
    int w = 0;
    for (int m = s_begin + GROUPS * q; m < min(s_end, s_begin + GROUPS * (q + 1)); ++m) w += bound[(size_t)blockIdx.z * nsrc + m];
    round_bound[q] = w;
  }
  __syncwarp();
  if (warp == MMA_WARP) tmem_alloc(smem_u32(tmem_slot), 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t sbase = smem_u32(smem);

  if (warp < GEN_WARPS) {
    // ---- digits of W: warpgroup g takes every second source (GROUPS = 2), thread = target row
    const int g = warp >> 2, row = threadIdx.x & (ROWS - 1);
    const int l = row0 + blockIdx.x * ROWS + row;
    const bool lvalid = l < row0 + nrows;
    const double xl = lvalid ? cx[l] : 0.0, yl = lvalid ? cy[l] : 0.0;
    bool ok = true;
    for (int q = 0; q < rounds && ok; ++q) {
      const int m = s_begin + GROUPS * q + g;
      PairSeed o;
      o.j0 = o.y0 = o.j1 = o.y1 = o.c = o.s = o.w = 0;
      if (lvalid && m < s_end && src0 + m != l) {
        const double dx = xl - cx[src0 + m], dy = yl - cy[src0 + m];
        const double r2 = fma(dx, dx, dy * dy);
        if (!pair_is_near(r2, pc)) pair_seed(dx, dy, r2, pc, stab, o);
      }
      PairState a;
      PairStep step;
      pair_start(o, a, step);
      for (int c = 0; c < chunks; ++c) {
        const int t = (q * chunks + c) * GROUPS + g;
        const int st = t % STAGES, lap = t / STAGES;
        // all lanes give up together: the others would wait for this one at the warp's barrier below
        if (lap > 0 && !__all_sync(0xffffffffu, mbar_wait(empty0 + 8 * st, (lap - 1) & 1))) {
          ok = false;
          break;
        }
        unsigned char* base = smem + st * STAGE + row * 16;
#pragma unroll 1
        for (int kg = 0; kg < KG && KG * c + kg < 2 * steps; ++kg) {
          uint32_t u[PL], v[PL], w[PL], z[PL];
          if (KG * c + kg <= p) {                  // orders 2 (KG c + kg) and the next
            int64_t pr[8];
            pair_two_orders(a, step, (int64_t)digit_bias<PL>(), pr);
            biased_digit_pairs<PL>(pr[0], pr[1], u);
            biased_digit_pairs<PL>(pr[2], pr[3], v);
            biased_digit_pairs<PL>(pr[4], pr[5], w);
            biased_digit_pairs<PL>(pr[6], pr[7], z);
          } else {
#pragma unroll
            for (int j = 0; j < PL; ++j) u[j] = v[j] = w[j] = z[j] = 0;
          }
#pragma unroll
          for (int j = 0; j < PL; ++j)
            *(uint4*)(base + j * A_PLANE + kg * A_KG) = make_uint4(u[j], v[j], w[j], z[j]);
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(full0 + 8 * st);
      }
    }
    if (!ok && lane == 0) atomicExch(err, 11);
  } else if (warp < MMA_WARP) {
    // ---- drain: warp d owns lanes 32 (d mod 4) .. + 31 and half of the columns
    const int d = warp - GEN_WARPS, quad = warp & 3, half = d >> 2;
    constexpr int HC = NPAD / 2;
    int64_t acc[HC];
#pragma unroll
    for (int i = 0; i < HC; ++i) acc[i] = 0;
    const uint32_t tb = tmem + ((uint32_t)(32 * quad) << 16) + half * HC;
    bool ok = true;
    for (int q = 0, group = 0; q < rounds; ++group) {
      int sum = 0;
      do sum += round_bound[q++];
      while (q < rounds && sum + round_bound[q] <= kExact);      // the issuing warp's groups
      ok = __all_sync(0xffffffffu, mbar_wait(accf, group & 1));
      if (!ok) break;
      tc_fence_after();
      if (six) drain_levels<NPAD, 5>(tb, acc);
      else drain_levels<NPAD, 6>(tb, acc);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acce);
    }
    if (ok) {
      const int row = blockIdx.x * ROWS + 32 * quad + lane;
      const int ex = scale_exponent(mb) - 48;      // unit of acc
      if (row < nrows && !(stat.count == 1 && row0 + row == stat.disc)) {
#pragma unroll
        for (int i = 0; i < HC; ++i) {
          const int col = half * HC + i;
          if (col < 2 * P)
            atomicAdd((double*)(ar + (size_t)row * P) + col, fixed_to_double(acc[i], ex));
        }
      }
    } else if (lane == 0) {
      atomicExch(err, 12);
    }
  } else {
    if (warp == MMA_WARP && lane == 0) {
      // ---- MMA issue
      bool ok = true;
      int t = 0, group = 0, sum = 0;
      for (int q = 0; q < rounds && ok; ++q) {
        const int w = round_bound[q];
        const bool start = q == 0 || sum + w > kExact;
        sum = start ? w : sum + w;
        if (start && q > 0) {
          mma_commit(accf);
          if (!mbar_wait(acce, group & 1)) {
            ok = false;
            break;
          }
          ++group;
          tc_fence_after();
        }
        for (int c = 0; c < GROUPS * chunks; ++c, ++t) {
          const int st = t % STAGES, lap = t / STAGES;
          if (!mbar_wait(full0 + 8 * st, lap & 1)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = sbase + st * STAGE;
          const int ksteps = min(2, steps - 2 * (c / GROUPS));
          for (int ks = 0; ks < ksteps; ++ks) {
            const bool first = start && c == 0 && ks == 0;
            if (six) issue_step<Tile, NPAD, 5>(tmem, sa, sa + A_BYTES, ks, first);
            else issue_step<Tile, NPAD, 6>(tmem, sa, sa + A_BYTES, ks, first);
          }
          mma_commit(empty0 + 8 * st);
        }
      }
      if (ok) mma_commit(accf);
      if (!ok) atomicExch(err, 13);
    } else if (warp == MMA_WARP + 1 && lane == 0) {
      // ---- copies of the X digits
      bool ok = true;
      constexpr uint32_t STEP = 2 * b_kg_bytes(NPAD);
      const size_t src_bytes = (size_t)steps * STEP;
      const unsigned char* ir = img + (size_t)blockIdx.z * nsrc * src_bytes;
      int t = 0;
      for (int q = 0; q < rounds && ok; ++q)
        for (int c = 0; c < chunks && ok; ++c)
          for (int g = 0; g < GROUPS; ++g, ++t) {
            const int st = t % STAGES, lap = t / STAGES;
            if (lap > 0 && !mbar_wait(empty0 + 8 * st, (lap - 1) & 1)) {
              ok = false;
              break;
            }
            const int m = min(s_begin + GROUPS * q + g, s_end - 1);
            const uint32_t bytes = min(2, steps - 2 * c) * STEP;
            mbar_expect_tx(full0 + 8 * st, bytes);
            bulk_load(sbase + st * STAGE + A_BYTES, ir + m * src_bytes + (size_t)c * 2 * STEP, bytes, full0 + 8 * st);
          }
      // copies still in flight end before the CTA does
      for (int s = max(0, t - STAGES); s < t && !ok; ++s) mbar_wait(full0 + 8 * (s % STAGES), (s / STAGES) & 1);
      if (!ok) atomicExch(err, 14);
    }
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == MMA_WARP) tmem_dealloc(tmem, 512);
}

// ---------------------------------------------------------------------------------------------
// Near pairs: k rho below pair_z_near (H_{2p} would leave the fixed-point range), from their list.
// ---------------------------------------------------------------------------------------------
// h_s, s = -2p..2p, of the pair offset (dx, dy); h points at s = 0.
__device__ __forceinline__ void pair_sequence(double dx, double dy, double k, int p, double2* h) {
  const double rho = hypot(dx, dy), z = k * rho, iz = 1.0 / z;
  const double2 e1 = make_double2(dx / rho, dy / rho);
  double2 hm = make_double2(j0(z), y0(z)), hq = make_double2(j1(z), y1(z)), eq = e1;
  h[0] = hm;
  for (int q = 1; q <= 2 * p; ++q) {
    h[q] = cmul(hq, eq);
    const double2 u = cmul(hq, make_double2(eq.x, -eq.y));
    h[-q] = (q & 1) ? make_double2(-u.x, -u.y) : u;
    const double f = 2.0 * q * iz;
    const double2 hn = make_double2(f * hq.x - hm.x, f * hq.y - hm.y);
    hm = hq;
    hq = hn;
    eq = cmul(eq, e1);
  }
}
// The sequences of every listed pair, once per layout: seq[pair][4p + 1]; zero for the candidates that
// the digit kernel takes (its own decision, pair_is_near).
__global__ void k_near_sequences(const double* __restrict__ cx, const double* __restrict__ cy,
                                 const int* __restrict__ tgt, const int* __restrict__ idx, int nnz, int p, double k,
                                 PairConsts pc, double2* __restrict__ seq) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nnz) return;
  const int l = tgt[e], m = idx[e];
  double2* h = seq + (size_t)e * (4 * p + 1) + 2 * p;
  const double dx = cx[l] - cx[m], dy = cy[l] - cy[m];
  if (pair_is_near(fma(dx, dx, dy * dy), pc)) {
    pair_sequence(dx, dy, k, p, h);
  } else {
    for (int q = -2 * p; q <= 2 * p; ++q) h[q] = make_double2(0.0, 0.0);
  }
}

// ---------------------------------------------------------------------------------------------
// The far pairs of the one disc whose coefficients are more than 16 times all others': its own row does not
// contain it, so the digits, which are cut relative to it, are too coarse there (one disc 1e8 larger: 6e-5
// of that row at 1500 discs).  Summed in FP64, a warp per 32 sources; without such a disc the CTAs return.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(32)
k_dominant_row(const double* __restrict__ cx, const double* __restrict__ cy, int n, int p, double k, PairConsts pc,
               const double2* __restrict__ xs, const RhsStats* __restrict__ stats, int row0, int nrows,
               double2* __restrict__ alpha) {
  __shared__ double2 seq[32][4 * LSMS_MAX_P + 1];
  const int P = 2 * p + 1, lane = threadIdx.x, r = blockIdx.y;
  const RhsStats s = stats[r];
  const int l = s.disc;
  if (s.count != 1 || s.maxbits >= kInfBits || l < row0 || l >= row0 + nrows) return;
  const int m0 = blockIdx.x * 32, m = m0 + lane;
  bool far = false;
  if (m < n && m != l) {
    const double dx = cx[l] - cx[m], dy = cy[l] - cy[m];
    far = !pair_is_near(fma(dx, dx, dy * dy), pc);
    if (far) pair_sequence(dx, dy, k, p, &seq[lane][2 * p]);
  }
  const unsigned mask = __ballot_sync(0xffffffffu, far);
  __syncwarp();
  if (lane >= P) return;
  double2 a = make_double2(0.0, 0.0);
  for (int i = 0; i < 32; ++i) {
    if (!(mask >> i & 1)) continue;
    const double2* b = xs + ((size_t)r * n + m0 + i) * P;
    for (int q = 0; q < P; ++q) a = cfma(seq[i][2 * p - lane + q], b[q], a);
  }
  double2* o = alpha + ((size_t)r * nrows + (l - row0)) * P + lane;
  atomicAdd(&o->x, a.x);
  atomicAdd(&o->y, a.y);
}

template <int NPAD>
void launch_digits(dim3 grid, cudaStream_t st, const lsms_ctx* c, const PairConsts& pc, const unsigned char* img,
                   const int* bound, int src0, int nsrc, int per_cta, int r0, const RhsStats* stats,
                   int row0, int nrows, double2* alpha, int* err) {
  static std::once_flag attr;
  std::call_once(attr, [] {
    cudaFuncSetAttribute(k_translate_digits<NPAD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)smem_bytes(NPAD));
  });
  k_translate_digits<NPAD><<<grid, THREADS, smem_bytes(NPAD), st>>>(
      c->d_cx, c->d_cy, c->n, c->p, pc, (const longlong2*)c->f64tc.d_table, img, bound, src0, nsrc, per_cta, r0,
      stats, row0, nrows, alpha, err);
}

constexpr size_t kImageBytes = (size_t)256 << 20;   // digits of X held at once
// p = 12: 96 discs 75 us from stored sequences and 86 as digits, 112 discs 101 and 87, 150 discs 155 and 89
constexpr int kMinDiscs = 96;
// mostly near pairs, p = 12: 320 discs (80 MB) 713 us stored and 732 on the FP64 pipe, 600 discs 2.27 and
// 2.40 ms, 1000 discs (780 MB) 7.05 and 6.52 ms: too little either way for the memory
constexpr double kStoreBytes = 64e6;
constexpr double kNearBytes = 8e9;                  // near sequences beside the digits

}  // namespace

void f64tc_free(lsms_ctx* c) {
  F64Tc& f = c->f64tc;
  void* ptrs[] = {f.d_table, f.d_seq};             // d_ptr and d_idx lie behind the table
  for (void* p : ptrs)
    if (p) cudaFree(p);
  f = F64Tc();
}

// Tables of the layout: `ptr`, `idx` list per target the sources within (1 + 1e-6) of the near
// distance (host arrays).  Layouts of fewer than kMinDiscs discs (not one full tile of rows) or of
// mostly near pairs (summed on the FP64 pipe either way) store the sequences of all their pairs if
// these take at most kStoreBytes (16 discs: 75 us with the sequences formed anew -> 11 us);
// larger ones, layouts for whose tables there is no memory and lengths below 1e-18 or above 1e18 keep
// k_translate_f64 and its symmetric form.
int f64tc_setup(lsms_ctx* c, const std::vector<int>& ptr, const std::vector<int>& idx) {
  f64tc_free(c);
  F64Tc& f = c->f64tc;
  const int n = c->n;
  if (n <= 0 || !tc_err_flag(c)) return LSMS_OK;
  // near and far pairs are told apart by squared distances in FP32, whose range these must not leave (in
  // any unit of length in use they do not)
  double reach = c->d;
  for (int j = 0; j < n; ++j) reach = std::max(reach, 2.0 * std::fabs(c->cx[j] - c->xc));
  if (!(pair_z_near(c->p) / c->k2 > 1e-18) || !(reach < 1e18)) return LSMS_OK;
  const double seq_bytes = (4 * c->p + 1) * (double)sizeof(double2);
  const bool digits = n >= kMinDiscs && (double)idx.size() <= 0.5 * n * (double)(n - 1) &&
                      (double)idx.size() * seq_bytes <= kNearBytes;
  const bool store = !digits && (double)n * (n - 1) * seq_bytes <= kStoreBytes;
  if (!digits && !store) return LSMS_OK;
  std::vector<int> all_ptr, all_idx;
  if (store) {
    all_ptr.resize(n + 1);
    for (int l = 0; l <= n; ++l) all_ptr[l] = l * (n - 1);
    for (int l = 0; l < n; ++l)
      for (int m = 0; m < n; ++m)
        if (m != l) all_idx.push_back(m);
  }
  const std::vector<int>&lp = store ? all_ptr : ptr, &li = store ? all_idx : idx;
  const long double pi = 3.14159265358979323846264338327950288L;
  std::vector<longlong2> tab(256);
  for (int i = 0; i < 256; ++i) {
    const long double a = 2 * pi * i / 256 - pi / 4, one = 4611686018427387904.0L;
    tab[i] = make_longlong2((long long)rintl(cosl(a) * one), (long long)rintl(sinl(a) * one));
  }
  const size_t nnz = li.size(), ne = nnz > 0 ? nnz : 1;
  std::vector<int> tgt(nnz);
  for (int l = 0; l < n; ++l)
    for (int e = lp[l]; e < lp[l + 1]; ++e) tgt[e] = l;
  // one allocation: table, list pointers, sources, targets
  const size_t bytes = TABLE_BYTES + ((size_t)(n + 1) + 2 * ne) * sizeof(int);
  if (device_alloc_optional(c, &f.d_table, bytes) != cudaSuccess) {
    f64tc_free(c);
    return LSMS_OK;
  }
  f.d_ptr = (int*)((unsigned char*)f.d_table + TABLE_BYTES);
  f.d_idx = f.d_ptr + n + 1;
  std::vector<unsigned char> host(bytes, 0);
  std::memcpy(host.data(), tab.data(), TABLE_BYTES);
  std::memcpy(host.data() + TABLE_BYTES, lp.data(), (n + 1) * sizeof(int));
  if (nnz) {
    std::memcpy(host.data() + TABLE_BYTES + (n + 1) * sizeof(int), li.data(), nnz * sizeof(int));
    std::memcpy(host.data() + TABLE_BYTES + (n + 1 + nnz) * sizeof(int), tgt.data(), nnz * sizeof(int));
  }
  copy_up(c, f.d_table, host.data(), bytes);
  f.nnz = (int)nnz;
  f.ready = true;
  f.digits = digits;
  return check_cuda(c, "f64tc_setup");
}

// The near sequences (63 MB at 5000 discs, p = 14) are stored when all-pairs FP64 translations can first
// run: not while every translation goes through boxes, nor in a mixed context that has had none
// (its solves come to them with their first FP64 residual).  They stay for the layout: an application
// captured before boxes were switched on refers to them.
int f64tc_sequences(lsms_ctx* c) {
  F64Tc& f = c->f64tc;
  const bool want = f.ready && f.nnz > 0 && (c->precision != LSMS_MIXED || f.used) &&
                    !(c->fmm.ready && c->fmm.scope == LSMS_FMM_ALL);
  if (!want || f.d_seq) return LSMS_OK;
  if (device_alloc_optional(c, &f.d_seq, (size_t)f.nnz * (4 * c->p + 1) * sizeof(double2)) != cudaSuccess) {
    f64tc_free(c);
    return LSMS_OK;
  }
  k_near_sequences<<<(f.nnz + 127) / 128, 128, 0, c->stream>>>(c->d_cx, c->d_cy, f.d_idx + f.nnz, f.d_idx, f.nnz,
                                                                c->p, c->k2,
                                                                pair_consts(c->k2, f.digits ? pair_z_near(c->p) : HUGE_VAL),
                                                                (double2*)f.d_seq);
  cudaStreamSynchronize(c->stream);
  return check_cuda(c, "f64tc_sequences");
}

bool f64tc_usable(const lsms_ctx* c) { return c->f64tc.ready && (c->f64tc.nnz == 0 || c->f64tc.d_seq); }

// alpha = rows row0 .. row0 + nrows - 1 of T xs, [nrhs][nrows][P].
int translate_f64_tc(lsms_ctx* c, int nrhs, const double2* xs, double2* alpha, cudaStream_t st, int row0, int nrows) {
  F64Tc& f = c->f64tc;
  const int n = c->n, p = c->p, P = c->P, npad = pad_columns(p), steps = k_steps(p);
  cudaMemsetAsync(alpha, 0, (size_t)nrhs * nrows * P * sizeof(double2), st);
  if (!f.digits) {
    // about 8 warps per SM
    if (f.nnz > 0) {
      ++c->f64_launches;
      const int splits = (int)std::max<long long>(1, std::min<long long>(n - 1, 152LL * 8 / std::max(1LL, (long long)nrows * nrhs)));
      launch_near_f64(n, p, nullptr, row0, nrows, splits, f.d_ptr, f.d_idx, (const double2*)f.d_seq, xs, nrhs, alpha, st);
    }
    return check_cuda(c, "translate_f64_tc");
  }
  const size_t src_bytes = (size_t)2 * steps * b_kg_bytes(npad);
  // the image holds whole right-hand sides if several fit, else a run of sources of one
  const int cap = (int)std::max<size_t>(1, kImageBytes / src_bytes);
  const int rb = std::max(1, std::min(nrhs, cap / n));
  int runs = (n + cap - 1) / cap;
  const int run = (n + runs - 1) / runs;
  runs = (n + run - 1) / run;
  const size_t img_bytes = (size_t)rb * std::min(run, n) * src_bytes;
  const size_t stat_bytes = ((size_t)nrhs * sizeof(RhsStats) + 255) & ~size_t(255);
  const size_t max_bytes = stat_bytes + (((size_t)nrhs * n * 8 + 255) & ~size_t(255));
  const size_t bound_bytes = ((size_t)rb * std::min(run, n) * sizeof(int) + 255) & ~size_t(255);
  // without memory for the image (or inside a capture that began before there was one): the FP64 pipe
  if (!ensure_optional(c, c->ws_f64tc, max_bytes + bound_bytes + img_bytes, st)) {
    launch_translate_f64(c->d_cx, c->d_cy, n, p, c->k2, xs, alpha, nrhs, st, row0, nrows);
    ++c->f64_launches;
    return check_cuda(c, "translate_f64");
  }
  RhsStats* stats = (RhsStats*)c->ws_f64tc.ptr;
  unsigned long long* dmax = (unsigned long long*)((unsigned char*)c->ws_f64tc.ptr + stat_bytes);
  int* bound = (int*)((unsigned char*)c->ws_f64tc.ptr + max_bytes);
  unsigned char* img = (unsigned char*)c->ws_f64tc.ptr + max_bytes + bound_bytes;
  int* err = tc_err_flag(c);
  cudaMemsetAsync(stats, 0, (size_t)nrhs * sizeof(RhsStats), st);
  k_disc_max<<<dim3((n + 7) / 8, nrhs), 256, 0, st>>>(xs, n, P, dmax, stats);
  k_large_discs<<<nrhs, 256, 0, st>>>(n, dmax, stats);
  const PairConsts pc = pair_consts(c->k2, pair_z_near(p));
  const int tiles = (nrows + ROWS - 1) / ROWS;
  for (int r0 = 0; r0 < nrhs; r0 += rb) {
    const int nr = std::min(rb, nrhs - r0);
    for (int s0 = 0; s0 < n; s0 += run) {
      const int ns = std::min(run, n - s0);
      c->f64_launches += 2;
      k_pack_digits<<<dim3(ns, nr), 256, 0, st>>>(xs, n, p, s0, r0, npad, 2 * steps, stats, img, bound);
      // source ranges: the fewest waves of 152 CTAs times the rounds of two sources of a CTA, plus
      // about two rounds of time per CTA for its start and end
      int best = 1;
      double cost = 1e300;
      const int max_split = std::min((ns + GROUPS - 1) / GROUPS, 152 * 8);
      for (int sp = (ns + MAX_SOURCES - 1) / MAX_SOURCES; sp <= max_split; ++sp) {
        const double waves = std::ceil((double)tiles * sp * nr / 152.0);
        const double cc = waves * (2.0 + std::ceil(std::ceil((double)ns / sp) / GROUPS));
        if (cc < cost * 0.999) {
          cost = cc;
          best = sp;
        }
      }
      const int per_cta = (((ns + best - 1) / best) + GROUPS - 1) / GROUPS * GROUPS;
      dim3 grid(tiles, (ns + per_cta - 1) / per_cta, nr);
#define LSMS_DG(NP) launch_digits<NP>(grid, st, c, pc, img, bound, s0, ns, per_cta, r0, stats, row0, nrows, alpha, err)
      if (npad == 32) LSMS_DG(32);
      else if (npad == 48) LSMS_DG(48);
      else LSMS_DG(64);
#undef LSMS_DG
    }
  }
  k_dominant_row<<<dim3((n + 31) / 32, nrhs), 32, 0, st>>>(c->d_cx, c->d_cy, n, p, c->k2, pc, xs, stats, row0, nrows,
                                                          alpha);
  c->f64_launches += 3 + (f.nnz > 0 ? 1 : 0);          // maxima, large discs, the dominant row, near pairs
  // lists cut so that the warps fill the chip (300 discs: 161 -> 107 us the translation, 1000: 478 -> 444)
  const int near_splits = (int)std::max<long long>(1, std::min<long long>(4, 152LL * 24 / std::max(1LL, (long long)nrows * nrhs)));
  if (f.nnz > 0)
    launch_near_f64(n, p, nullptr, row0, nrows, near_splits, f.d_ptr, f.d_idx, (const double2*)f.d_seq, xs, nrhs, alpha, st);
  return check_cuda(c, "translate_f64_tc");
}
