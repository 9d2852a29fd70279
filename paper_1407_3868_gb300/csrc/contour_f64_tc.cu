// FP64 contour contractions on the tensor cores: the aggregate G = E_agg . x (Thm 5.2 / Eq. "invfft")
// and the disaggregate alpha += E_dis . V (Lemma 5.1 / Eq. "JA2") as products of 48-bit fixed-point
// operands (digits_tc.cuh), for layouts whose tables fill the chip.
//
// A complex row (a_r0, a_i0, a_r1, ...) meets the real embedding of the right operand (column Re: b_r,
// -b_i; column Im: b_i, b_r).  E_agg is scaled by a power of two per row (a contour node decays
// with Re gamma y).  E_dis is scaled per column: V grows with lambda^order where E_dis decays, so the
// column scales move onto V, whose columns (orders) are then scaled by their largest element.  What
// is rounded away is below 2^-48 of the largest term of a sum; the tables' own FP64 phases
// (lambda x up to 1e5) are off by more.
//
// The FP64 tables are read once and cut into digits on the way to shared memory (a lane takes one
// complex element, a warp one 8-row x 4-element core matrix: 64 contiguous bytes per row from
// memory, 32 distinct banks on the store).  The bound is that read (164 MB for 5000 discs and 1024
// nodes: 24 us at the measured copy rate); the two products take 102 and 113 us there, on the FP64
// pipe (tiled products in shared memory) they took 2.5 ms each.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "digits_tc.cuh"
#include "lsms_internal.h"
#include "lsms_ops.h"

namespace {

constexpr int CK = 16;                          // complex K elements of a stage
constexpr int GEN_WARPS = 8;
constexpr int THREADS = (GEN_WARPS + DRAIN_WARPS + 2) * 32;
constexpr int MAX_K = 8192;                     // complex K elements per CTA (64-bit sums)
constexpr size_t zsmem_bytes(int npad) { return (size_t)STAGES * stage_bytes(npad) + 256; }

__device__ __forceinline__ unsigned long long mag_bits(double2 v) {
  const unsigned long long a = (unsigned long long)__double_as_longlong(v.x) & 0x7fffffffffffffffull;
  const unsigned long long b = (unsigned long long)__double_as_longlong(v.y) & 0x7fffffffffffffffull;
  return a > b ? a : b;
}

// Largest |Re|, |Im| of every row (one warp each) of a [rows][cols] table.
__global__ void k_row_max(const double2* __restrict__ a, int rows, int cols, unsigned long long* __restrict__ out) {
  const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (r >= rows) return;
  unsigned long long m = 0;
  for (int c = lane; c < cols; c += 32) m = max(m, mag_bits(a[(size_t)r * cols + c]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) out[r] = m;
}
// The same of every column; grid.y ranges of rows, out zeroed.
__global__ void k_col_max(const double2* __restrict__ a, int rows, int cols, int per, unsigned long long* __restrict__ out) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cols) return;
  unsigned long long m = 0;
  const int r1 = min(rows, (int)(blockIdx.y + 1) * per);
  for (int r = blockIdx.y * per; r < r1; ++r) m = max(m, mag_bits(a[(size_t)r * cols + c]));
  if (m) atomicMax(out + c, m);
}
// exponents (0 for an empty row); bad is set for a non-finite table
__global__ void k_exponents(const unsigned long long* __restrict__ bits, int count, int* __restrict__ e, int* __restrict__ bad) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const unsigned long long b = bits[i];
  if (b >= kInfBits) atomicExch(bad, 1);
  e[i] = b == 0 || b >= kInfBits ? 0 : scale_exponent(b);
}

// Largest |Re|, |Im| of every (right-hand side, order) of b [r][K][P], element k times 2^kexp[k].
__global__ void k_order_max(const double2* __restrict__ b, int K, int P, const int* __restrict__ kexp, int per,
                            unsigned long long* __restrict__ out) {
  const int q = threadIdx.x & 31, r = blockIdx.y;
  if (q >= P) return;
  const int k1 = min(K, (int)(blockIdx.x + 1) * per);
  unsigned long long m = 0;
  for (int k = blockIdx.x * per + (threadIdx.x >> 5); k < k1; k += blockDim.x >> 5) {
    unsigned long long v = mag_bits(b[((size_t)r * K + k) * P + q]);
    if (kexp && v && v < kInfBits)
      v = (unsigned long long)__double_as_longlong(scalbn(__longlong_as_double((long long)v), kexp[k]));
    m = max(m, v);
  }
  if (m) atomicMax(out + r * 32 + q, m);
}

// Digits of the right operand: per right-hand side [stage][K group][plane][column][8 K values].
__global__ void k_pack_columns(const double2* __restrict__ b, int K, int P, int r0, int stages, int npad,
                               const int* __restrict__ kexp, const unsigned long long* __restrict__ maxbits,
                               unsigned char* __restrict__ img) {
  const int r = r0 + blockIdx.y, half = npad / 2;
  uint4* dst = (uint4*)(img + (size_t)blockIdx.y * stages * KG * b_kg_bytes(npad));
  const int total = stages * KG * half;
  for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < total; it += gridDim.x * blockDim.x) {
    const int kg = it / half, q = it - kg * half;
    uint32_t wr[PL][4], wi[PL][4];
    const unsigned long long mb = q < P ? maxbits[r * 32 + q] : 0;
    const bool live = mb != 0 && mb < kInfBits;
    const int sh = live ? 47 - scale_exponent(mb) : 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = 4 * kg + i;
      long long re = 0, im = 0;
      if (live && k < K) {
        const double2 v = b[((size_t)r * K + k) * P + q];
        const int s = sh + (kexp ? kexp[k] : 0);
        re = llrint(scalbn(v.x, s));
        im = llrint(scalbn(v.y, s));
      }
      uint32_t u[PL], v2[PL];
      digit_pairs(re << 16, -im << 16, u);
      digit_pairs(im << 16, re << 16, v2);
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

// v 2^(63 - e) as an integer (|v| <= 0.99 2^e), truncated; what is below its unit is dropped.
__device__ __forceinline__ int64_t to_q63(double v, int e) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const int ex = (int)((hi >> 20) & 0x7ff);
  const uint64_t m = ((uint64_t)((hi & 0xfffff) | 0x100000) << 32 | lo) << 10;
  const int shift = min(1022 - ex + e, 63);
  int64_t q = (int64_t)(m >> shift);
  if (ex == 0) q = 0;
  return (int32_t)hi < 0 ? -q : q;
}

// C[r][m][q] += sum_k A[m][k] B[r][k][q].  ROWEXP: A scaled by 2^-aexp[m], else by 2^-aexp[k] (the
// inverse is in the image).  grid: (row tiles, K ranges, right-hand sides).
template <int NPAD, bool ROWEXP>
__global__ void __launch_bounds__(THREADS, 1)
k_zgemm_digits(const double2* __restrict__ A, int M, int K, const int* __restrict__ aexp,
               const unsigned char* __restrict__ img, int stages, int per_cta, int P, int r0,
               const unsigned long long* __restrict__ maxbits, double2* __restrict__ C, int* __restrict__ err) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int STAGE = stage_bytes(NPAD), LMAX = 6;
  uint64_t* bars = (uint64_t*)(smem + STAGES * STAGE);   // full[S], empty[S], acc_full, acc_empty
  uint32_t* tmem_slot = (uint32_t*)(bars + 2 * STAGES + 2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = r0 + blockIdx.z, m0 = blockIdx.x * ROWS;
  const int t_begin = blockIdx.y * per_cta, nt = min(stages - t_begin, per_cta);
  if (nt <= 0) return;
  const int groups = (nt + DRAIN - 1) / DRAIN;
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
  __syncwarp();
  if (warp == GEN_WARPS + DRAIN_WARPS) tmem_alloc(smem_u32(tmem_slot), 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t sbase = smem_u32(smem);

  if (warp < GEN_WARPS) {
    // ---- digits of A: the warps of group g take every second stage, 16 core matrices each
    const int g = warp >> 2, w = warp & 3;
    const int rr = lane >> 2, ke = lane & 3;       // row and complex element in a core matrix
    bool ok = true;
    for (int t = g; t < nt; t += 2) {
      const int st = t % STAGES, round = t / STAGES;
      const int kb = (t_begin + t) * CK + ke;
#pragma unroll 1
      for (int h = 0; h < 2 && ok; ++h) {          // 8 core matrices at a time: rows 32 w + 16 h ..
        double2 v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int row = m0 + 32 * w + 16 * h + 8 * (i & 1) + rr, k = kb + 4 * (i >> 1);
          v[i] = row < M && k < K ? __ldg(A + (size_t)row * K + k) : make_double2(0.0, 0.0);
        }
        if (h == 0 && round > 0 && !mbar_wait(empty0 + 8 * st, (round - 1) & 1)) {
          ok = false;
          break;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int row = 32 * w + 16 * h + 8 * (i & 1) + rr, k = kb + 4 * (i >> 1);
          const int e = ROWEXP ? (m0 + row < M ? aexp[m0 + row] : 0) : (k < K ? aexp[k] : 0);
          uint32_t u[PL];
          digit_pairs(to_q63(v[i].x, e), to_q63(v[i].y, e), u);
          unsigned char* d = smem + st * STAGE + (i >> 1) * A_KG + row * 16 + ke * 4;
#pragma unroll
          for (int j = 0; j < PL; ++j) *(uint32_t*)(d + j * A_PLANE) = u[j];
        }
      }
      if (!__all_sync(0xffffffffu, ok)) {
        ok = false;
        break;
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(full0 + 8 * st);
    }
    if (!ok && lane == 0) atomicExch(err, 21);
  } else if (warp < GEN_WARPS + DRAIN_WARPS) {
    // ---- drain: warp d owns lanes 32 (d mod 4) .. + 31 and half of the columns
    const int d = warp - GEN_WARPS, quad = warp & 3, half = d >> 2;
    constexpr int HC = NPAD / 2;
    int64_t acc[HC];
#pragma unroll
    for (int i = 0; i < HC; ++i) acc[i] = 0;
    const uint32_t tb = tmem + ((uint32_t)(32 * quad) << 16) + half * HC;
    bool ok = true;
    for (int q = 0; q < groups; ++q) {
      ok = __all_sync(0xffffffffu, mbar_wait(accf, q & 1));
      if (!ok) break;
      tc_fence_after();
      drain_levels<NPAD, LMAX>(tb, acc);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acce);
    }
    if (ok) {
      const int row = m0 + 32 * quad + lane;
      if (row < M) {
        const int re = ROWEXP ? aexp[row] : 0;
#pragma unroll
        for (int i = 0; i < HC; ++i) {
          const int col = half * HC + i;
          if (col < 2 * P) {
            const unsigned long long mb = maxbits[r * 32 + (col >> 1)];
            const int ex = mb && mb < kInfBits ? re + scale_exponent(mb) - 48 : 0;   // unit of acc
            double v = fixed_to_double(acc[i], ex);
            if (mb >= kInfBits) v = __longlong_as_double(0x7ff8000000000000ll);
            if (mb) atomicAdd((double*)(C + ((size_t)r * M + row) * P) + col, v);
          }
        }
      }
    } else if (lane == 0) {
      atomicExch(err, 22);
    }
  } else if (warp == GEN_WARPS + DRAIN_WARPS) {
    // ---- MMA issue
    if (lane == 0) {
      bool ok = true;
      for (int t = 0; t < nt; ++t) {
        const int st = t % STAGES, round = t / STAGES, q = t / DRAIN;
        const bool start = t % DRAIN == 0;
        if ((start && q > 0 && !mbar_wait(acce, (q - 1) & 1)) || !mbar_wait(full0 + 8 * st, round & 1)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t sa = sbase + st * STAGE;
        for (int ks = 0; ks < KG / 2; ++ks)
          issue_step<NPAD, LMAX>(tmem, sa, sa + A_BYTES, ks, start && ks == 0);
        mma_commit(empty0 + 8 * st);
        if (t % DRAIN == DRAIN - 1 || t == nt - 1) mma_commit(accf);
      }
      if (!ok) atomicExch(err, 23);
    }
    __syncwarp();
  } else {
    // ---- copies of the image
    if (lane == 0) {
      bool ok = true;
      constexpr uint32_t BYTES = KG * b_kg_bytes(NPAD);
      const unsigned char* ir = img + ((size_t)blockIdx.z * stages + t_begin) * BYTES;
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

template <int NPAD, bool ROWEXP>
void launch_digits(dim3 grid, cudaStream_t st, const double2* A, int M, int K, const int* aexp,
                   const unsigned char* img, int stages, int per_cta, int P, int r0,
                   const unsigned long long* maxbits, double2* C, int* err) {
  static std::once_flag attr;
  std::call_once(attr, [] {
    cudaFuncSetAttribute(k_zgemm_digits<NPAD, ROWEXP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)zsmem_bytes(NPAD));
  });
  k_zgemm_digits<NPAD, ROWEXP><<<grid, THREADS, zsmem_bytes(NPAD), st>>>(A, M, K, aexp, img, stages, per_cta, P, r0,
                                                                         maxbits, C, err);
}

constexpr size_t kImageBytes = (size_t)128 << 20;

}  // namespace

void zgemm_free(lsms_ctx* c) {
  ZgemmTc& z = c->zgemm;
  if (z.d_exp) cudaFree(z.d_exp);
  if (z.ws.ptr) cudaFree(z.ws.ptr);
  z = ZgemmTc();
}

// Row exponents of E_agg and column exponents of E_dis.
int zgemm_setup(lsms_ctx* c) {
  zgemm_free(c);
  ZgemmTc& z = c->zgemm;
  const int n = c->n, rows = 2 * c->ns;
  if ((double)rows * n < kZgemmMinTable || !tc_err_flag(c)) return LSMS_OK;
  // one allocation: exponents, then the maxima they come from
  const size_t eb = ((size_t)2 * rows * sizeof(int) + 15) & ~size_t(15), bb = (size_t)2 * rows * 8 + 16;
  if (cudaMalloc((void**)&z.d_exp, eb + bb) != cudaSuccess) {
    cudaGetLastError();
    zgemm_free(c);
    return LSMS_OK;                                // the FP64 pipe then (launch_zgemm_direct)
  }
  unsigned long long* bits = (unsigned long long*)((unsigned char*)z.d_exp + eb);
  int* bad = (int*)(bits + 2 * rows);
  cudaMemsetAsync(bits, 0, bb, c->stream);
  k_row_max<<<(rows + 7) / 8, 256, 0, c->stream>>>(c->d_eagg, rows, n, bits);
  const int per = std::max(1, (n + 63) / 64);
  k_col_max<<<dim3((rows + 127) / 128, (n + per - 1) / per), 128, 0, c->stream>>>(c->d_edis, n, rows, per, bits + rows);
  k_exponents<<<(2 * rows + 255) / 256, 256, 0, c->stream>>>(bits, 2 * rows, z.d_exp, bad);
  int h = 0;
  cudaMemcpyAsync(&h, bad, sizeof(int), cudaMemcpyDeviceToHost, c->stream);
  cudaStreamSynchronize(c->stream);
  z.ready = h == 0;
  return check_cuda(c, "zgemm_setup");
}

// C[r][M][P] += table . B for the aggregate (M = 2 N_S, K = n) or the disaggregate (M = n, K = 2 N_S).
int zgemm_f64(lsms_ctx* c, bool agg, int nrhs, const double2* B, double2* C, cudaStream_t st) {
  ZgemmTc& z = c->zgemm;
  const int P = c->P, M = agg ? 2 * c->ns : c->n, K = agg ? c->n : 2 * c->ns;
  const double2* A = agg ? c->d_eagg : c->d_edis;
  if (!z.ready) {
    launch_zgemm_direct(A, M, K, B, C, P, nrhs, st);
    return LSMS_OK;
  }
  const int npad = pad_columns(c->p), stages = (K + CK - 1) / CK;
  const int max_stages = (std::max(c->n, 2 * c->ns) + CK - 1) / CK;
  const size_t sb = (size_t)KG * b_kg_bytes(npad);
  const int rb = (int)std::max<size_t>(1, std::min<size_t>(nrhs, kImageBytes / (max_stages * sb)));
  const size_t mbytes = ((size_t)nrhs * 32 * 8 + 255) & ~size_t(255);
  if (ensure(c, z.ws, mbytes + (size_t)rb * max_stages * sb)) {   // no memory for the image
    c->err.clear();
    launch_zgemm_direct(A, M, K, B, C, P, nrhs, st);
    return check_cuda(c, "zgemm_f64");
  }
  unsigned long long* maxbits = (unsigned long long*)z.ws.ptr;
  unsigned char* img = (unsigned char*)z.ws.ptr + mbytes;
  const int* kexp = agg ? nullptr : z.d_exp + 2 * c->ns;
  const int* aexp = agg ? z.d_exp : kexp;
  int* err = tc_err_flag(c);
  cudaMemsetAsync(maxbits, 0, (size_t)nrhs * 32 * 8, st);
  const int per = std::max(8, (K + 127) / 128);
  k_order_max<<<dim3((K + per - 1) / per, nrhs), 256, 0, st>>>(B, K, P, kexp, per, maxbits);
  const int mt = (M + ROWS - 1) / ROWS;
  for (int r0 = 0; r0 < nrhs; r0 += rb) {
    const int nr = std::min(rb, nrhs - r0);
    const int items = stages * KG * (npad / 2);
    k_pack_columns<<<dim3(std::min((items + 127) / 128, 1024), nr), 128, 0, st>>>(B, K, P, r0, stages, npad, kexp,
                                                                                maxbits, img);
    // K ranges: the fewest rounds of 152 CTAs times the stages of a CTA, plus a start and an end worth
    // about six stages
    int best = 1;
    double cost = 1e300;
    for (int sp = (stages + MAX_K / CK - 1) / (MAX_K / CK); sp <= std::min(stages, 152 * 4); ++sp) {
      const double cc = std::ceil((double)mt * sp * nr / 152.0) * (6.0 + std::ceil((double)stages / sp));
      if (cc < cost * 0.999) {
        cost = cc;
        best = sp;
      }
    }
    const int per_cta = (stages + best - 1) / best;
    dim3 grid(mt, (stages + per_cta - 1) / per_cta, nr);
#define LSMS_ZG(NP)                                                                                              \
  (agg ? launch_digits<NP, true>(grid, st, A, M, K, aexp, img, stages, per_cta, P, r0, maxbits, C, err)          \
       : launch_digits<NP, false>(grid, st, A, M, K, aexp, img, stages, per_cta, P, r0, maxbits, C, err))
    if (npad == 32) LSMS_ZG(32);
    else if (npad == 48) LSMS_ZG(48);
    else LSMS_ZG(64);
#undef LSMS_ZG
  }
  return check_cuda(c, "zgemm_f64");
}
