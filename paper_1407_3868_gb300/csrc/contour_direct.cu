// FP64 contour contractions of small tables (below 1.5e5 complex elements) on the FP64 pipe: a warp per
// output row, lane = output order, the table element a broadcast and the right operand's row a
// coalesced load.  What bounds them is latency, so the aggregate, the order sums, the reflection and
// the disaggregate's right operand are one kernel (a warp per contour node), and K is cut so that the
// products spread over the chip.  16 discs, 256 nodes:
// 15 and 8 us for the two kernels, 32 us the whole reflected coupling with its neighbours (98 us with
// tiled products in shared memory).
#include <algorithm>

#include "c64.cuh"
#include "lsms_internal.h"
#include "lsms_ops.h"

namespace {

// sum_{k0 <= k < k1} a[k] b[k][lane] over the P orders (idle lanes repeat the last one); ORDER: b[order[k]],
// nothing where that is negative (a[k] is zero there)
template <bool ORDER>
__device__ __forceinline__ double2 row_sum(const double2* __restrict__ a, const double2* __restrict__ b,
                                           const int* __restrict__ order, int P, int q, int k0, int k1) {
  double rr = 0.0, ii = 0.0, ri = 0.0, ir = 0.0;
#pragma unroll 4
  for (int k = k0; k < k1; ++k) {
    const double2 u = __ldg(a + k), v = __ldg(b + (size_t)(ORDER ? max(0, __ldg(order + k)) : k) * P + q);
    rr = fma(u.x, v.x, rr);
    ii = fma(u.y, v.y, ii);
    ri = fma(u.x, v.y, ri);
    ir = fma(u.y, v.x, ir);
  }
  return make_double2(rr - ii, ri + ir);
}

// C[r][m][q] += sum_k A[m][k] B[r][k][q]; a warp per (row, K range, right-hand side).  ORDER: B[r] has n
// rows, taken in this order.
template <bool ORDER>
__global__ void __launch_bounds__(128)
k_zgemm_direct(const double2* __restrict__ A, int M, int K, const double2* __restrict__ B, double2* __restrict__ C,
               int P, int per, const int* __restrict__ order, int n) {
  const int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31, r = blockIdx.y;
  const int chunks = (K + per - 1) / per, m = w / chunks;
  if (m >= M) return;
  const int k0 = (w - m * chunks) * per;
  const double2 s = row_sum<ORDER>(A + (size_t)m * K, B + (size_t)r * (ORDER ? n : K) * P, order, P,
                                   min(lane, P - 1), k0, min(K, k0 + per));
  if (lane < P) {
    double* o = (double*)(C + ((size_t)r * M + m) * P + lane);
    atomicAdd(o, s.x);
    atomicAdd(o + 1, s.y);
  }
}

// Per contour node (warp): G = E_agg x for its two rows, the order sums P+, Q-, the reflection and
// V = U sigma (k_node_stage with the aggregate inside).
__global__ void __launch_bounds__(128)
k_node_direct(int ns, int n, int P, const double2* __restrict__ eagg, const double2* __restrict__ xs,
              const double2* __restrict__ fagg, const double2* __restrict__ refl, const double2* __restrict__ udis,
              double2* __restrict__ V) {
  const int v = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31, r = blockIdx.y;
  if (v >= ns) return;
  const int q = min(lane, P - 1);
  const double2* b = xs + (size_t)r * n * P;
  double2 gp = row_sum<false>(eagg + (size_t)v * n, b, nullptr, P, q, 0, n);
  double2 gm = row_sum<false>(eagg + (size_t)(ns + v) * n, b, nullptr, P, q, 0, n);
  gp = lane < P ? cmul(fagg[(size_t)v * P + q], gp) : make_double2(0.0, 0.0);
  gm = lane < P ? cmul(fagg[(size_t)(ns + v) * P + q], gm) : make_double2(0.0, 0.0);
  const double2 Pp = warp_sum(gp), Qm = warp_sum(gm);
  const double2 sp = cadd(cmul(refl[4 * v], Pp), cmul(refl[4 * v + 1], Qm));
  const double2 sm = cadd(cmul(refl[4 * v + 2], Pp), cmul(refl[4 * v + 3], Qm));
  if (lane < P) {
    V[((size_t)r * 2 * ns + v) * P + lane] = cmul(udis[(size_t)v * P + lane], sp);
    V[((size_t)r * 2 * ns + ns + v) * P + lane] = cmul(udis[(size_t)(ns + v) * P + lane], sm);
  }
}

}  // namespace

void launch_zgemm_direct(const double2* A, int M, int K, const double2* B, double2* C, int P, int nrhs,
                         cudaStream_t st, const int* order, int n) {
  if (M == 0 || K == 0 || nrhs == 0) return;
  // about 16 warps per SM, at least 16 elements of K each
  const int chunks = (int)std::max<long long>(1, std::min<long long>((K + 15) / 16, 152LL * 16 / std::max(1LL, (long long)M * nrhs)));
  const int per = (K + chunks - 1) / chunks, nc = (K + per - 1) / per;
  const long long warps = (long long)M * nc;
  const int wpc = small_block(warps * nrhs);
  const dim3 grid((unsigned)((warps + wpc - 1) / wpc), nrhs);
  if (order) k_zgemm_direct<true><<<grid, 32 * wpc, 0, st>>>(A, M, K, B, C, P, per, order, n);
  else k_zgemm_direct<false><<<grid, 32 * wpc, 0, st>>>(A, M, K, B, C, P, per, nullptr, 0);
}

void launch_node_direct(int ns, int n, int P, int nrhs, const double2* eagg, const double2* xs, const double2* fagg,
                        const double2* refl, const double2* udis, double2* V, cudaStream_t st) {
  const int wpc = small_block((long long)ns * nrhs);
  k_node_direct<<<dim3((ns + wpc - 1) / wpc, nrhs), 32 * wpc, 0, st>>>(ns, n, P, eagg, xs, fagg, refl, udis, V);
}
