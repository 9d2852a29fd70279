// FP64 sums over listed pairs whose Hankel sequences are stored (Sec. 3.2 Lemma 3.1): the near pairs
// of the tensor-core translation and every pair of short layouts (translate_f64_tc.cu), the same- and
// adjacent-box pairs of the translation through boxes (fmm.cu).
#pragma once

#include <cuda_runtime.h>

#include "lsms_internal.h"

namespace {

// alpha^l += sum over the sources listed for row t, l = perm[t] (perm: targets in box order; rows row0 ..
// row0 + nrows - 1 of alpha otherwise): one warp per (target, right-hand side), lane = output order.
// The sequences are read where they lie (a window of P consecutive values per source order, in L1
// after the first; the lists of 5000 discs at p = 14 take 63 MB, in L2 between applications), so the
// kernel needs no shared memory and enough warps share an SM to keep its FP64 pipe busy: four
// independent FMAs per order and warp.  The near pairs of 5000 discs: 2.80 ms with the sequences formed
// anew in shared memory (one CTA per SM) -> 0.51 ms (its 8 M warp FMAs take 0.44 ms of the pipe); the
// adjacent boxes of 20,000 discs (472,000 pairs): 4.65 -> 3.2 ms (2.95 ms of the pipe).
// Short layouts, all of whose pairs are stored, cut the lists into `splits` parts that add atomically:
// 16 discs are 240 warps of one pair instead of 16 warps of 15.
__global__ void __launch_bounds__(128)
k_near_f64(int n, int p, const int* __restrict__ perm, int row0, int nrows, int splits,
           const int* __restrict__ ptr, const int* __restrict__ idx, const double2* __restrict__ seq,
           const double2* __restrict__ xs, double2* __restrict__ alpha) {
  const int P = 2 * p + 1, lane = threadIdx.x & 31, r = blockIdx.y;
  const int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), part = w % splits;
  const int t = row0 + w / splits;
  if (t >= row0 + nrows) return;
  const int l = perm ? perm[t] : t, len = ptr[t + 1] - ptr[t];
  const int e0 = ptr[t] + (int)((long long)len * part / splits), e1 = ptr[t] + (int)((long long)len * (part + 1) / splits);
  const double2* xr = xs + (size_t)r * n * P;
  const int nu = min(lane, P - 1);                       // idle lanes repeat the last order
  double rr = 0.0, ii = 0.0, ri = 0.0, ir = 0.0;
  for (int e = e0; e < e1; ++e) {
    const double2* h = seq + (size_t)e * (4 * p + 1) + 2 * p - nu;
    const double2* b = xr + (size_t)idx[e] * P;
#pragma unroll 4
    for (int q = 0; q < P; ++q) {
      const double2 hv = __ldg(h + q), bv = __ldg(b + q);
      rr = fma(hv.x, bv.x, rr);
      ii = fma(hv.y, bv.y, ii);
      ri = fma(hv.x, bv.y, ri);
      ir = fma(hv.y, bv.x, ir);
    }
  }
  if (lane < P) {
    double2* o = alpha + ((size_t)r * nrows + (l - row0)) * P + lane;
    if (splits == 1) {
      *o = make_double2(o->x + (rr - ii), o->y + (ri + ir));
    } else if (e1 > e0) {
      atomicAdd(&o->x, rr - ii);
      atomicAdd(&o->y, ri + ir);
    }
  }
}


inline void launch_near_f64(int n, int p, const int* perm, int row0, int nrows, int splits, const int* ptr,
                            const int* idx, const double2* seq, const double2* xs, int nrhs, double2* alpha,
                            cudaStream_t st) {
  if (nrows <= 0 || nrhs <= 0) return;
  const long long warps = (long long)nrows * splits;
  const int per = small_block(warps * nrhs);   // warps per CTA
  k_near_f64<<<dim3((unsigned)((warps + per - 1) / per), nrhs), 32 * per, 0, st>>>(n, p, perm, row0, nrows, splits,
                                                                                         ptr, idx, seq, xs, alpha);
}

}  // namespace
