// FP64 contour contractions on the tensor cores: the aggregate G = E_agg . x (Thm 5.2 / Eq. "invfft")
// and the disaggregate alpha += E_dis . V (Lemma 5.1 / Eq. "JA2") as products of 56-bit fixed-point
// operands (digits_tc.cuh, seven digits, levels 0..6), for layouts whose tables fill the chip.
//
// A complex row (a_r0, a_i0, a_r1, ...) meets the real embedding of the right operand (column Re: b_r,
// -b_i; column Im: b_i, b_r).  A fixed-point operand keeps its bits below one scale, and the tables
// fall with e^{-Re gamma t} over the distance t of a disc from an interface (Re gamma up to 160, t
// from 0.3 to 1.7 in the usual layer): one scale per row of E_agg, or per column of E_dis, would leave
// nothing of the deep discs there.  So the discs are taken in order of depth, in classes graded by
// their distance from the nearer interface (depth_classes), and every class has scales of its own:
//   aggregate:    the sum over a class's discs scales E_agg by its largest element in (class, node), x by
//                 its largest in (class, order), and is added to G by itself;
//   disaggregate: for the targets of a class E_dis is scaled per node (V grows with lambda^order where
//                 E_dis decays, so the inverse scale moves onto V), and V then per order; V is packed
//                 once for every class.
// What is rounded away is 2^-54 of (largest element) x (largest coefficient) of the class.  Worst row of
// the reflected coupling against 64 bits, orders unscaled, 1500 discs: 1.9e-11 on random coefficients and
// 1.2e-11 on coefficients of one size in every order, as the FP64 pipe's sums (the phases lambda x
// carry that); with one scale per row and six digits it was 9.7e-10 and 3.5e-5.  A single node where only
// the deepest disc of a class has coefficients loses e^{Re gamma (t - t_min)} of these bits: lsms_aggregate
// and lsms_disaggregate, which show single nodes, sum on the FP64 pipe.
//
// The FP64 tables are read once and cut into digits on the way to shared memory (a lane takes one
// complex element, a warp one 8-row x 4-element core matrix: 64 contiguous bytes per row from
// memory, 32 distinct banks on the store; E_agg's columns are stored in order of depth).  The whole reflected coupling of 5000 discs and 1024 nodes
// takes 0.28 ms (0.27 ms with one scale per row and six digits, 5.1 ms on the FP64 pipe; the tables'
// two reads are 0.05 ms), of 1000 discs and 512 nodes 101 us (FP64 pipe: 546 us), of 20,000 discs 0.82 ms (20 ms).
// The products are bound by the conversion (ALU pipe at half its peak) and the waits between it, the MMAs
// and the drains.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "digits_tc.cuh"
#include "lsms_internal.h"
#include "lsms_ops.h"

namespace {

using Tile = DigitTile<7, 2>;                   // a stage: one MMA step, 16 real K values
constexpr int PL = Tile::PL, KG = Tile::KG, A_PLANE = Tile::A_PLANE, A_BYTES = Tile::A_BYTES;
constexpr int LMAX = 6;
constexpr int STAGES = 5;
constexpr int CK = 8;                           // complex K elements of a stage
constexpr int DRAIN = 12;                       // stages per drain: 192 K values, on which level 4 is exact
constexpr int GEN_WARPS = 8;
constexpr int THREADS = (GEN_WARPS + DRAIN_WARPS + 2) * 32;
constexpr int MAX_NT = 2048;                    // stages per CTA
constexpr int CLASSES = 32;                     // at most; 8 in the usual layer
constexpr double kClassRatio = 1.36;            // of a class's distances from the nearer interface
constexpr int kNan = 1 << 14, kNone = -kNan;    // column exponents of a non-finite and of a zero column
constexpr int kEmpty = -4096;                   // 2^kEmpty times any double is zero
constexpr int kRoom = 8;                        // order maxima are kept 2^-8 smaller: scaled by E they stay finite
constexpr size_t zsmem_bytes(int npad) {
  return (size_t)STAGES * Tile::stage_bytes(npad) + MAX_NT + CLASSES * 64 * sizeof(short) + 256;
}

__device__ __forceinline__ unsigned long long mag_bits(double2 v) {
  const unsigned long long a = (unsigned long long)__double_as_longlong(v.x) & 0x7fffffffffffffffull;
  const unsigned long long b = (unsigned long long)__double_as_longlong(v.y) & 0x7fffffffffffffffull;
  return a > b ? a : b;
}

// out[r][e] = a[r][kidx[e]] (zero where that is negative), e < ld: the columns of E_agg in their classes.
__global__ void k_order_columns(const double2* __restrict__ a, int rows, int cols, const int* __restrict__ kidx, int ld,
                                double2* __restrict__ out) {
  const long long total = (long long)rows * ld;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const long long r = i / ld;
    const int k = kidx[i - r * ld];
    out[i] = k >= 0 ? a[r * cols + k] : make_double2(0.0, 0.0);
  }
}
// Largest |Re|, |Im| of every (class, row) of that table [rows][ld], one warp each; the class's columns are
// start[c] .. start[c + 1] - 1.
__global__ void k_row_max(const double2* __restrict__ a, int rows, int ld, const int* __restrict__ start,
                          unsigned long long* __restrict__ out) {
  const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31, c = blockIdx.y;
  if (r >= rows) return;
  unsigned long long m = 0;
  for (int e = start[c] + lane; e < start[c + 1]; e += 32) m = max(m, mag_bits(a[(size_t)r * ld + e]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) out[(size_t)c * rows + r] = m;
}
// The same of every (class, column) of E_dis, the class's rows kidx[start[c]] .. kidx[start[c + 1] - 1], negative
// entries are padding; out zeroed, grid.z parts of the class.
__global__ void k_col_max(const double2* __restrict__ a, int cols, const int* __restrict__ kidx,
                          const int* __restrict__ start, unsigned long long* __restrict__ out) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x, c = blockIdx.y;
  if (v >= cols) return;
  unsigned long long m = 0;
  for (int e = start[c] + blockIdx.z; e < start[c + 1]; e += gridDim.z) {
    const int k = kidx[e];
    if (k >= 0) m = max(m, mag_bits(a[(size_t)k * cols + v]));
  }
  if (m) atomicMax(out + (size_t)c * cols + v, m);
}
// exponents, kEmpty for a row or column that is all zero (e^{-Re gamma t} has underflowed): the right operand
// meets nothing there, and must not count among its order's largest; bad is set for a non-finite table
__global__ void k_exponents(const unsigned long long* __restrict__ bits, int count, int* __restrict__ e, int* __restrict__ bad) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const unsigned long long b = bits[i];
  if (b >= kInfBits) atomicExch(bad, 1);
  e[i] = b == 0 ? kEmpty : b >= kInfBits ? 0 : scale_exponent(b);
}

// Largest |Re|, |Im| of every (right-hand side, class, order) of b [r][K][P], times 2^-kRoom.
// Aggregate (kexp null): over the class's discs.  Disaggregate: over all nodes, element k times
// 2^kexp[class][k].
__global__ void __launch_bounds__(256)
k_order_max(const double2* __restrict__ b, int K, int P, const int* __restrict__ kidx,
                            const int* __restrict__ start, const int* __restrict__ kexp,
                            unsigned long long* __restrict__ out) {
  __shared__ unsigned long long part[8][32];
  const int q = threadIdx.x & 31, r = blockIdx.y, c = blockIdx.z;
  const int w = threadIdx.x >> 5, step = gridDim.x * 8;
  const int e0 = kexp ? 0 : start[c], e1 = kexp ? K : start[c + 1];
  unsigned long long m = 0;
  for (int e = e0 + blockIdx.x * 8 + w; e < e1 && q < P; e += step) {
    const int k = kexp ? e : kidx[e];
    if (k < 0) continue;
    unsigned long long v = mag_bits(b[((size_t)r * K + k) * P + q]);
    if (v && v < kInfBits)
      v = (unsigned long long)__double_as_longlong(
          scalbn(__longlong_as_double((long long)v), (kexp ? kexp[(size_t)c * K + k] : 0) - kRoom));
    m = max(m, v);
  }
  part[w][q] = m;                                  // one update per CTA: the addresses are few
  __syncthreads();
  if (w > 0) return;
  for (int i = 1; i < 8; ++i) m = max(m, part[i][q]);
  if (m) atomicMax(out + ((size_t)r * gridDim.z + c) * 32 + q, m);
}

// v 2^(63 - e) as an integer (|v| <= 0.99 2^e), truncated; what is below its unit is dropped.
__device__ __forceinline__ int64_t to_q63(double v, int e) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const int ex = (int)((hi >> 20) & 0x7ff);
  const uint64_t m = ((uint64_t)((hi & 0xfffff) | 0x100000) << 32 | lo) << 10;
  const int shift = min(max(1022 - ex + e, 0), 63);   // a zero may come with any e
  int64_t q = (int64_t)(m >> shift);
  if (ex == 0) q = 0;
  return (int32_t)hi < 0 ? -q : q;
}

// Digits of the right operand, [r][image][stage][K group][plane][column][8 K values].  Aggregate: one
// image, its K order kidx, the scales of the stage's class.  Disaggregate (kexp): an image per class,
// K order the nodes', the inverse of E's scales on top.
__global__ void k_pack_columns(const double2* __restrict__ b, int K, int P, int r0, int stages, int npad, int classes,
                               const int* __restrict__ kidx, const unsigned char* __restrict__ scls,
                               const int* __restrict__ kexp, const unsigned long long* __restrict__ maxbits,
                               unsigned char* __restrict__ img) {
  const int r = r0 + blockIdx.y, half = npad / 2;
  uint4* dst = (uint4*)(img + ((size_t)blockIdx.y * gridDim.z + blockIdx.z) * stages * KG * Tile::b_kg_bytes(npad));
  const int total = stages * KG * half;
  for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < total; it += gridDim.x * blockDim.x) {
    const int kg = it / half, q = it - kg * half;
    const int c = kexp ? blockIdx.z : scls[kg / KG];
    uint32_t wr[PL][4], wi[PL][4];
    const unsigned long long mb = q < P ? maxbits[((size_t)r * classes + c) * 32 + q] : 0;
    const bool live = mb != 0 && mb < kInfBits;
    const int ex = live ? scale_exponent(mb) + kRoom : 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int kp = 4 * kg + i, k = kexp ? (kp < K ? kp : -1) : kidx[kp];
      int64_t re = 0, im = 0;
      if (live && k >= 0) {
        const double2 v = b[((size_t)r * K + k) * P + q];
        const int e = ex - (kexp ? kexp[(size_t)c * K + k] : 0);
        re = to_q63(v.x, e);
        im = to_q63(v.y, e);
      }
      uint32_t u[PL], v2[PL];
      digit_pairs<PL>(re, -im, u);
      digit_pairs<PL>(im, re, v2);
#pragma unroll
      for (int j = 0; j < PL; ++j) {
        wr[j][i] = u[j];
        wi[j][i] = v2[j];
      }
    }
#pragma unroll
    for (int j = 0; j < PL; ++j) {
      uint4* d = dst + ((size_t)kg * PL + j) * npad + 2 * q;
      d[0] = make_uint4(wr[j][0], wr[j][1], wr[j][2], wr[j][3]);
      d[1] = make_uint4(wi[j][0], wi[j][1], wi[j][2], wi[j][3]);
    }
  }
}

// Sum of one group's levels in units of level 5 (2^-54 of the product of the scales).
__device__ __forceinline__ int64_t level_sum(const uint32_t* f) {
  const int lo = __float2int_rn(__uint_as_float(f[5])) + ((__float2int_rn(__uint_as_float(f[6])) + 128) >> 8);
  int64_t v = mad_wide(__float2int_rn(__uint_as_float(f[4])), 1 << 8, lo);
  v = mad_wide(__float2int_rn(__uint_as_float(f[3])), 1 << 16, v);
  v = mad_wide(__float2int_rn(__uint_as_float(f[2])), 1 << 24, v);
  // |level 0| <= 192 2^14, |level 1| <= 2 192 2^14: the high word below stays under 2^30
  const int hi = __float2int_rn(__uint_as_float(f[1])) + __float2int_rn(__uint_as_float(f[0])) * 256;
  return v + shl(hi, 32);
}

// End of the group of stages that starts at t: the next class, DRAIN stages, or nt.
__device__ __forceinline__ int group_end(const unsigned char* cls, int t, int nt) {
  int e = t + 1;
  while (e < nt && e - t < DRAIN && cls[e] == cls[t]) ++e;
  return e;
}

// C[r][m][q] += sum_k A[m][k] B[r][k][q].  AGG: rows m = the table's, its K columns in their classes, A scaled by
// 2^-aexp[class of the stage][m].  Else rows m = kidx[tile.y + i], i < tile.z, of class tile.x, K order
// the nodes', A scaled by 2^-aexp[class][k] (the inverse is in the image).  grid: (row tiles, K ranges,
// right-hand sides); shared memory fits one CTA per SM.
template <int NPAD, bool AGG>
__global__ void __launch_bounds__(THREADS, 1)
k_zgemm_digits(const double2* __restrict__ A, int M, int K, const int* __restrict__ kidx,
               const unsigned char* __restrict__ scls, const int4* __restrict__ tiles, int classes,
               const int* __restrict__ aexp, const unsigned char* __restrict__ img, int stages, int per_cta, int P,
               int r0, const unsigned long long* __restrict__ maxbits, double2* __restrict__ C,
               int* __restrict__ err) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int STAGE = Tile::stage_bytes(NPAD);
  unsigned char* cls = smem + STAGES * STAGE;                  // class of every stage of this CTA
  short* colx = (short*)(cls + MAX_NT);                        // [class][column]: exponent of the column's scale
  uint64_t* bars = (uint64_t*)(colx + CLASSES * 64);           // full[S], empty[S], acc_full, acc_empty
  uint32_t* tmem_slot = (uint32_t*)(bars + 2 * STAGES + 2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = r0 + blockIdx.z;
  const int t_begin = blockIdx.y * per_cta, nt = min(stages - t_begin, per_cta);
  if (nt <= 0) return;
  const int4 tile = AGG ? make_int4(0, 0, 0, 0) : tiles[blockIdx.x];
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * STAGES, accf = full0 + 16 * STAGES, acce = accf + 8;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full0 + 8 * s, 5);                 // four converting warps and the copy
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(accf, 1);
    mbar_init(acce, DRAIN_WARPS);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int t = threadIdx.x; t < nt; t += THREADS) cls[t] = AGG ? scls[t_begin + t] : (unsigned char)tile.x;
  for (int i = threadIdx.x; i < classes * NPAD; i += THREADS) {
    const int c = i / NPAD, col = i - c * NPAD;
    int e = kNone;
    if (col < 2 * P) {
      const unsigned long long mb = maxbits[((size_t)r * classes + c) * 32 + (col >> 1)];
      e = mb == 0 ? kNone : mb >= kInfBits ? kNan : scale_exponent(mb) + kRoom;
    }
    colx[i] = (short)e;
  }
  __syncwarp();
  if (warp == GEN_WARPS + DRAIN_WARPS) tmem_alloc(smem_u32(tmem_slot), 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t sbase = smem_u32(smem);

  if (warp < GEN_WARPS) {
    // ---- digits of A: the warps of group g take every second stage, 8 core matrices each: rows 32 w + 8 j + rr,
    // complex elements ke and ke + 4
    const int g = warp >> 2, w = warp & 3;
    const int rr = lane >> 2, ke = lane & 3;
    const double2* rp[4];
    int er[4], m[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int row = 32 * w + 8 * j + rr;
      if (AGG) m[j] = (int)blockIdx.x * ROWS + row < M ? (int)blockIdx.x * ROWS + row : -1;
      else m[j] = row < tile.z ? kidx[tile.y + row] : -1;
      rp[j] = A + (size_t)max(m[j], 0) * K;
      er[j] = 0;
    }
    auto k_at = [&](int t, int h) {
      const int kp = (t_begin + t) * CK + 4 * h + ke;
      return kp < K ? kp : -1;
    };
    int cur = -1;
    bool ok = true;
    for (int t = g; t < nt; t += 2) {
      const int st = t % STAGES, round = t / STAGES;
      double2 v[8];
      int ek[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k = k_at(t, h);
        ek[h] = !AGG && k >= 0 ? aexp[(size_t)tile.x * K + k] : 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) v[4 * h + j] = m[j] >= 0 && k >= 0 ? __ldg(rp[j] + k) : make_double2(0.0, 0.0);
      }
      if (AGG && cls[t] != cur) {
        cur = cls[t];
#pragma unroll
        for (int j = 0; j < 4; ++j) er[j] = m[j] >= 0 ? aexp[(size_t)cur * M + m[j]] : 0;
      }
      if (round > 0 && !__all_sync(0xffffffffu, mbar_wait(empty0 + 8 * st, (round - 1) & 1))) {
        ok = false;
        break;
      }
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int e = AGG ? er[j] : ek[h];
          uint32_t u[PL];
          digit_pairs<PL>(to_q63(v[4 * h + j].x, e), to_q63(v[4 * h + j].y, e), u);
          unsigned char* d = smem + st * STAGE + h * A_KG + (32 * w + 8 * j + rr) * 16 + ke * 4;
#pragma unroll
          for (int q = 0; q < PL; ++q) *(uint32_t*)(d + q * A_PLANE) = u[q];
        }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(full0 + 8 * st);
    }
    if (!ok && lane == 0) atomicExch(err, 21);
  } else if (warp < GEN_WARPS + DRAIN_WARPS) {
    // ---- drain: warp d owns lanes 32 (d mod 4) .. + 31 and half of the columns; every group is added to C
    const int d = warp - GEN_WARPS, quad = warp & 3, half = d >> 2;
    constexpr int HC = NPAD / 2;
    const uint32_t tb = tmem + ((uint32_t)(32 * quad) << 16) + half * HC;
    const int i = 32 * quad + lane;
    int m = -1;
    if (AGG) m = (int)blockIdx.x * ROWS + i < M ? (int)blockIdx.x * ROWS + i : -1;
    else if (i < tile.z) m = kidx[tile.y + i];
    double* out = (double*)(C + ((size_t)r * M + max(m, 0)) * P);
    bool ok = true;
    for (int t = 0, q = 0; t < nt; ++q) {
      const int c = cls[t];
      t = group_end(cls, t, nt);
      const int re = AGG && m >= 0 ? aexp[(size_t)c * M + m] : 0;
      ok = __all_sync(0xffffffffu, mbar_wait(accf, q & 1));
      if (!ok) break;
      tc_fence_after();
      int64_t acc[HC];
#pragma unroll
      for (int cb = 0; cb < HC / 4; ++cb) {
        uint32_t f[LMAX + 1][4];
        load_levels<NPAD, LMAX>(tb + 4 * cb, f);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          uint32_t e[LMAX + 1];
#pragma unroll
          for (int L = 0; L <= LMAX; ++L) e[L] = f[L][j];
          acc[4 * cb + j] = level_sum(e);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acce);
      if (m >= 0)
#pragma unroll
        for (int j = 0; j < HC; ++j) {
          const int ce = colx[c * NPAD + half * HC + j];
          if (ce == kNone) continue;
          const double v = ce == kNan ? __longlong_as_double(0x7ff8000000000000ll) : fixed_to_double(acc[j], re + ce - 54);
          atomicAdd(out + half * HC + j, v);
        }
    }
    if (!ok && lane == 0) atomicExch(err, 22);
  } else if (warp == GEN_WARPS + DRAIN_WARPS) {
    // ---- MMA issue
    if (lane == 0) {
      bool ok = true;
      for (int t = 0, q = 0; t < nt && ok; ++q) {
        const int t0 = t, t1 = group_end(cls, t, nt);
        if (q > 0 && !mbar_wait(acce, (q - 1) & 1)) {
          ok = false;
          break;
        }
        for (; t < t1; ++t) {
          const int st = t % STAGES, round = t / STAGES;
          if (!mbar_wait(full0 + 8 * st, round & 1)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = sbase + st * STAGE;
          issue_step<Tile, NPAD, LMAX>(tmem, sa, sa + A_BYTES, 0, t == t0);
          mma_commit(empty0 + 8 * st);
        }
        if (ok) mma_commit(accf);
      }
      if (!ok) atomicExch(err, 23);
    }
    __syncwarp();
  } else {
    // ---- copies of the image
    if (lane == 0) {
      bool ok = true;
      constexpr uint32_t BYTES = KG * Tile::b_kg_bytes(NPAD);
      const size_t image = AGG ? blockIdx.z : (size_t)blockIdx.z * classes + tile.x;
      const unsigned char* ir = img + (image * stages + t_begin) * BYTES;
      int t = 0;
      for (; t < nt; ++t) {
        const int st = t % STAGES, round = t / STAGES;
        if (round > 0 && !mbar_wait(empty0 + 8 * st, (round - 1) & 1)) {
          ok = false;
          break;
        }
        mbar_expect_tx(full0 + 8 * st, BYTES);
        bulk_load(sbase + st * STAGE + A_BYTES, ir + (size_t)t * BYTES, BYTES, full0 + 8 * st);
      }
      for (int s = max(0, t - STAGES); s < t && !ok; ++s) mbar_wait(full0 + 8 * (s % STAGES), (s / STAGES) & 1);
      if (!ok) atomicExch(err, 24);
    }
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == GEN_WARPS + DRAIN_WARPS) tmem_dealloc(tmem, 512);
}

struct Launch {
  dim3 grid;
  cudaStream_t st;
  const double2 *A, *B;
  double2* C;
  int M, K, stages, per_cta, r0;
  const int* aexp;
  const unsigned char* img;
  const unsigned long long* maxbits;
};
template <int NPAD, bool AGG>
void launch_digits(const lsms_ctx* c, const Launch& l, int* err) {
  static std::once_flag attr;
  std::call_once(attr, [] {
    cudaFuncSetAttribute(k_zgemm_digits<NPAD, AGG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)zsmem_bytes(NPAD));
  });
  const ZgemmTc& z = c->zgemm;
  k_zgemm_digits<NPAD, AGG><<<l.grid, THREADS, zsmem_bytes(NPAD), l.st>>>(
      l.A, l.M, l.K, c->d_eorder, z.d_scls, (const int4*)z.d_tiles, z.classes, l.aexp, l.img, l.stages, l.per_cta, c->P,
      l.r0, l.maxbits, l.C, err);
}

constexpr size_t kImageBytes = (size_t)128 << 20;

// The discs in order of depth, cut into classes evenly in the logarithm of the distance from the nearer
// interface, for either half of the layer: a term of order s falls with about the s-th power of the distance, so
// that a class's discs differ by its ratio to that power.  Discs 0.3 to 1.7 below the top of a layer of 2
// make 8 classes (ratio 1.35); errors of 6, 8 and 16 are the same there, and fewer classes leave fewer
// partly filled row tiles (200 discs, 2048 nodes: the reflected coupling 191 us with 16, 137 with 8).
// list: the classes' discs, each padded with -1 to a multiple of CK; start: classes + 1 positions.
void depth_classes(const lsms_ctx* c, std::vector<int>& list, std::vector<int>& start) {
  const int n = c->n;
  const double mid = 0.5 * c->d;
  double t0 = mid;
  for (int j = 0; j < n; ++j) t0 = std::min(t0, std::min(-c->cy[j], c->cy[j] + c->d));
  t0 = std::max(t0, 1e-6 * mid);
  const double top = std::log(mid / t0);
  const int count = 2 * std::min(CLASSES / 2, std::max(1, (int)std::ceil(top / std::log(kClassRatio))));
  std::vector<std::vector<int>> cl(count);
  for (int j = 0; j < n; ++j) {
    const double t = -c->cy[j], b = c->cy[j] + c->d, s = std::log(std::max(t0, std::min(t, b)) / t0);
    const double u = top > 0.0 ? 0.5 * (t <= b ? s : 2.0 * top - s) / top : 0.0;       // 0 .. 1 from top to bottom
    cl[std::min(count - 1, std::max(0, (int)(u * count)))].push_back(j);
  }
  list.clear();
  start.assign(1, 0);
  for (const std::vector<int>& v : cl) {
    if (v.empty()) continue;
    list.insert(list.end(), v.begin(), v.end());
    while (list.size() % CK) list.push_back(-1);
    start.push_back((int)list.size());
  }
}

inline size_t aligned(size_t bytes) { return (bytes + 255) & ~size_t(255); }

}  // namespace

void zgemm_free(lsms_ctx* c) {
  ZgemmTc& z = c->zgemm;
  if (z.d_exp) cudaFree(z.d_exp);
  z = ZgemmTc();
}

// The classes and the exponents of both tables in every class.
int zgemm_setup(lsms_ctx* c) {
  zgemm_free(c);
  ZgemmTc& z = c->zgemm;
  const int n = c->n, rows = 2 * c->ns;
  if ((double)rows * n < kZgemmMinTable || !tc_err_flag(c)) return LSMS_OK;
  std::vector<int> list, start;
  depth_classes(c, list, start);
  const int classes = (int)start.size() - 1;
  std::vector<unsigned char> scls(list.size() / CK);
  std::vector<int4> tiles;
  int widest = 0;
  for (int q = 0; q < classes; ++q) {
    for (int e = start[q]; e < start[q + 1]; e += CK) scls[e / CK] = (unsigned char)q;
    int count = start[q + 1] - start[q];
    widest = std::max(widest, count);
    while (list[start[q] + count - 1] < 0) --count;
    for (int i = 0; i < count; i += ROWS) tiles.push_back(make_int4(q, start[q] + i, std::min(ROWS, count - i), 0));
  }
  // one allocation: the exponents of E_agg and E_dis, the lists, then the maxima the exponents come from
  const size_t per = (size_t)classes * rows;
  const size_t be = aligned(2 * per * sizeof(int)), bs = aligned(scls.size()), bt = aligned(tiles.size() * sizeof(int4)),
               bc = aligned(start.size() * sizeof(int));
  const size_t lists = bs + bt + bc, bm = 2 * per * 8 + 16;
  const int ld = (int)list.size();
  double2* ordered = nullptr;
  int* order = nullptr;
  if (device_alloc_optional(c, (void**)&z.d_exp, be + lists + bm) != cudaSuccess ||
      device_alloc_optional(c, (void**)&ordered, (size_t)rows * ld * sizeof(double2)) != cudaSuccess ||
      device_alloc_optional(c, (void**)&order, ld * sizeof(int)) != cudaSuccess) {
    if (ordered) cudaFree(ordered);
    zgemm_free(c);
    return LSMS_OK;                                // the FP64 pipe then (launch_zgemm_direct)
  }
  // E_agg's columns class by class: gathered where they lie, its product took 246 instead of 103 us at 5000 discs
  copy_up(c, order, list.data(), ld * sizeof(int));
  k_order_columns<<<152 * 16, 256, 0, c->stream>>>(c->d_eagg, rows, n, order, ld, ordered);
  cudaStreamSynchronize(c->stream);
  cudaFree(c->d_eagg);
  c->d_eagg = ordered;
  c->d_eorder = order;
  c->eagg_ld = ld;
  unsigned char* at = (unsigned char*)z.d_exp + be;
  z.d_scls = at;
  z.d_tiles = at + bs;
  z.d_start = (int*)(at + bs + bt);
  std::vector<unsigned char> host(lists, 0);
  std::memcpy(host.data(), scls.data(), scls.size());
  std::memcpy(host.data() + bs, tiles.data(), tiles.size() * sizeof(int4));
  std::memcpy(host.data() + bs + bt, start.data(), start.size() * sizeof(int));
  unsigned long long* bits = (unsigned long long*)(at + lists);
  int* bad = (int*)(bits + 2 * per);
  copy_up(c, at, host.data(), lists);
  cudaMemsetAsync(bits, 0, bm, c->stream);
  k_row_max<<<dim3((rows + 7) / 8, classes), 256, 0, c->stream>>>(c->d_eagg, rows, ld, z.d_start, bits);
  k_col_max<<<dim3((rows + 127) / 128, classes, std::min(64, (widest + 63) / 64)), 128, 0, c->stream>>>(
      c->d_edis, rows, order, z.d_start, bits + per);
  k_exponents<<<(int)((2 * per + 255) / 256), 256, 0, c->stream>>>(bits, (int)(2 * per), z.d_exp, bad);
  int h = 0;
  cudaMemcpyAsync(&h, bad, sizeof(int), cudaMemcpyDeviceToHost, c->stream);
  cudaStreamSynchronize(c->stream);
  z.classes = classes;
  z.stages = (int)scls.size();
  z.tiles = (int)tiles.size();
  z.ready = h == 0;
  return check_cuda(c, "zgemm_setup");
}

void aggregate_direct(lsms_ctx* c, int nrhs, const double2* B, double2* G, cudaStream_t st) {
  launch_zgemm_direct(c->d_eagg, 2 * c->ns, c->eagg_ld, B, G, c->P, nrhs, st, c->d_eorder, c->n);
}

// C[r][M][P] += table . B for the aggregate (M = 2 N_S, K = the discs) or the disaggregate (M = n, K = 2 N_S).
int zgemm_f64(lsms_ctx* c, bool agg, int nrhs, const double2* B, double2* C, cudaStream_t st) {
  ZgemmTc& z = c->zgemm;
  Launch l;
  l.st = st;
  l.A = agg ? c->d_eagg : c->d_edis;
  l.B = B;
  l.C = C;
  l.M = agg ? 2 * c->ns : c->n;
  l.K = agg ? c->eagg_ld : 2 * c->ns;
  ++c->f64_launches;                                 // the direct product or the order maxima
  auto direct = [&] {
    if (agg) aggregate_direct(c, nrhs, B, C, st);
    else launch_zgemm_direct(l.A, l.M, l.K, B, C, c->P, nrhs, st);
    return check_cuda(c, "zgemm_f64");
  };
  if (!z.ready) return direct();
  const int npad = pad_columns(c->p), dis_stages = (2 * c->ns + CK - 1) / CK;
  l.stages = agg ? z.stages : dis_stages;
  const int images = agg ? 1 : z.classes;
  const size_t sb = (size_t)KG * Tile::b_kg_bytes(npad);
  // the workspace holds either product's images of as many right-hand sides as fit kImageBytes
  const size_t one = sb * std::max(z.stages, z.classes * dis_stages);
  const int rb = (int)std::max<size_t>(1, std::min<size_t>(nrhs, kImageBytes / one));
  const size_t mbytes = aligned((size_t)nrhs * z.classes * 32 * 8);
  if (!ensure_optional(c, c->ws_zgemm, mbytes + rb * one, st)) return direct();   // as in translate_f64_tc
  unsigned long long* maxbits = (unsigned long long*)c->ws_zgemm.ptr;
  unsigned char* img = (unsigned char*)c->ws_zgemm.ptr + mbytes;
  l.maxbits = maxbits;
  l.img = img;
  l.aexp = z.d_exp + (agg ? 0 : (size_t)z.classes * 2 * c->ns);
  const int* kexp = agg ? nullptr : l.aexp;
  int* err = tc_err_flag(c);
  cudaMemsetAsync(maxbits, 0, (size_t)nrhs * z.classes * 32 * 8, st);
  const int rows = agg ? c->n : l.K, mean = agg ? l.K / z.classes : l.K;       // rows of B, and of a class
  k_order_max<<<dim3(std::max(1, std::min(64, mean / 16)), nrhs, z.classes), 256, 0, st>>>(
      B, rows, c->P, c->d_eorder, z.d_start, kexp, maxbits);
  const int mt = agg ? (l.M + ROWS - 1) / ROWS : z.tiles;
  for (l.r0 = 0; l.r0 < nrhs; l.r0 += rb) {
    const int nr = std::min(rb, nrhs - l.r0);
    const int items = l.stages * KG * (npad / 2);
    c->f64_launches += 2;
    k_pack_columns<<<dim3(std::min((items + 127) / 128, 1024), nr, images), 128, 0, st>>>(
        B, rows, c->P, l.r0, l.stages, npad, z.classes, c->d_eorder, z.d_scls, kexp, maxbits, img);
    // K ranges: the fewest rounds of 152 CTAs times the stages of a CTA, plus a start and an end worth
    // about twelve stages
    int best = 1;
    double cost = 1e300;
    const int least = (l.stages + MAX_NT - 1) / MAX_NT;
    for (int sp = least; sp <= std::max(least, std::min(l.stages, 152 * 4)); ++sp) {
      const double cc = std::ceil((double)mt * sp * nr / 152.0) * (12.0 + std::ceil((double)l.stages / sp));
      if (cc < cost * 0.999) {
        cost = cc;
        best = sp;
      }
    }
    l.per_cta = (l.stages + best - 1) / best;
    l.grid = dim3(mt, (l.stages + l.per_cta - 1) / l.per_cta, nr);
#define LSMS_ZG(NP) (agg ? launch_digits<NP, true>(c, l, err) : launch_digits<NP, false>(c, l, err))
    if (npad == 32) LSMS_ZG(32);
    else if (npad == 48) LSMS_ZG(48);
    else LSMS_ZG(64);
#undef LSMS_ZG
  }
  return check_cuda(c, "zgemm_f64");
}
