// trmv's row sums (op(A)'s rows contiguous) on small triangles, in one launch: one cluster of 8 or 16 blocks.
//
// x is overwritten by the result, so nothing may be written before every block has read x.  The tile kernel leaves its sums to a second
// launch for that reason; here every block of the only cluster copies x to its shared memory and meets the others at a cluster barrier
// before it writes.  A warp has four neighbouring rows, its lanes along the columns, four packs (eight elements off 16-byte boundaries) of
// each row in flight.
//
// Bound by latency: the launch, x, the matrix through 16 SMs and the cluster barrier.  This product repeated, us, in two launches / so:
// float n = 64 4.4 / 2.8, 256 4.4 / 3.4, 400 4.6 / 3.8, 512 4.4 / 4.0; double 64 4.4 / 3.1, 200 5.2 / 3.7, 256 4.4 / 3.7, 300 4.5 / 5.1; off 16-byte
// boundaries float 128 4.5 / 2.7, 401 4.4 / 4.0, 601 5.0 / 6.1, double 401 4.7 / 4.5, 601 5.0 / 6.8.  The lines (limit()) lie where a copy and both
// products of a pass, the column sums in a launch of their own as before, are equal: float 400 10.8 / 9.7, 512 9.5 / 9.8, 294 (off) 10.6 / 11.3, double 200 11.0 / 9.3, 256 10.2 / 10.1, 359 (off) 10.8 / 11.9.
#pragma once

#include "level2.cuh"

namespace b2 {
namespace ts {

constexpr int kMaxCluster = 16, kRows = 4;
constexpr int kMaxN = kMaxCluster * kWarps * kRows;
template <typename T>
constexpr int limit(bool aligned) {
  static_assert(kMaxN >= 416, "four rows for each warp");
  return sizeof(T) == 4 ? (aligned ? 416 : 256) : 240;
}

// V: elements of a pack (1 off 16-byte boundaries).
template <typename T, int V, int TRI, bool UNIT>
__global__ void __launch_bounds__(kThreads) trmv_small_kernel(const T* __restrict__ a, int64_t lda, int n, T* x, int64_t incx) {
  cluster_arrive();
  grid_dep_wait();
  grid_dep_launch();
  __shared__ __align__(16) T xs[kMaxN + 4];
  constexpr int kPacks = V == 1 ? 8 : 4;  // of a row, in flight
  using P = Pack<T, V>;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int i = tid; i < (n + 3) / 4 * 4; i += kThreads) xs[i] = i < n ? x[i * incx] : T(0);
  __syncthreads();
  cluster_wait();  // (every block is running)
  __syncwarp();
  cluster_arrive();  // this block has read x
  const int i0 = ((int)cluster_rank() * kWarps + warp) * kRows;  // this warp's rows: i0 ..
  T sum = T(0);
  if (i0 < n) {  // (the same for a whole warp)
    const int lo = TRI == TRI_UPPER ? i0 / V * V : 0, hi = TRI == TRI_LOWER ? min(n, i0 + kRows) : n;
    T acc[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) acc[r] = T(0);
    for (int c0 = lo; c0 < hi; c0 += 32 * V * kPacks) {
      P m[kRows][kPacks];
#pragma unroll
      for (int u = 0; u < kPacks; ++u) {
        const int j = c0 + (u * 32 + lane) * V;
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
          const T* q = a + (int64_t)(i0 + r) * lda + j;
          const bool row = i0 + r < n && (TRI == TRI_UPPER ? j + V - 1 >= i0 + r : j <= i0 + r);
          m[r][u] = ld_nc_if<T, V>(q, row && j + V <= n);
          if (V > 1 && row && j < n && j + V > n) {
#pragma unroll
            for (int e = 0; e < V; ++e) m[r][u].v[e] = ld_el_if<T>(q + e, j + e < n);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kPacks; ++u) {
        const int j = c0 + (u * 32 + lane) * V;
#pragma unroll
        for (int e = 0; e < V; ++e) {
          if (j + e >= n) continue;
          const T xj = xs[j + e];
#pragma unroll
          for (int r = 0; r < kRows; ++r) {
            const int d = j + e - (i0 + r);
            const T v = UNIT && d == 0 ? T(1) : m[r][u].v[e];
            if (TRI == TRI_UPPER ? d >= 0 : d <= 0) acc[r] = v * xj + acc[r];
          }
        }
      }
    }
    sum = multi_group_sum<32, kRows>(acc, lane);  // of row lane / 8
  }
  __syncwarp();
  cluster_wait();  // every block has read x
  constexpr int LPR = 32 / kRows;
  const int i = i0 + lane / LPR;
  if (lane % LPR == 0 && i < n) B2_STORE(x + i * incx, sum);
}

// False (nothing launched) where the device has no clusters of that size.
template <typename T, int V, int TRI, bool UNIT>
static bool launch(const Launch& l, const L2Args<T>& q) {
  auto kern = trmv_small_kernel<T, V, TRI, UNIT>;
  const unsigned blocks = q.rows <= 8 * kWarps * kRows ? 8 : kMaxCluster;
  if (blocks > 8) {
    static signed char allowed[64];  // per device: 0 not asked yet
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    if (allowed[dev] == 0) {
      int fits = 0;
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = blocks;
      at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
      cfg.gridDim = dim3(blocks);
      cfg.blockDim = dim3(kThreads);
      cfg.attrs = at;
      cfg.numAttrs = 1;
      const bool ok = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                      cudaOccupancyMaxActiveClusters(&fits, kern, &cfg) == cudaSuccess && fits > 0;
      (void)cudaGetLastError();
      allowed[dev] = ok ? 1 : -1;
    }
    if (allowed[dev] < 0) return false;
  }
  launch_clusters(kern, blocks, blocks, dim3(kThreads), 0, l.stream, q.a, q.lda, (int)q.rows, q.y, q.incy);
  return true;
}
template <typename T, int TRI>
static int run(const Launch& l, const L2Args<T>& q, bool unit, bool* handled) {
  constexpr int V = VecLen<T>::value;
  *handled = false;
  const bool al = aligned_to(q.a, 16) && q.lda % V == 0;
  if (q.rows > (knob(kKnobGather) >= 2 ? kMaxN : limit<T>(al))) return B2_STATUS_OK;
  if (al) *handled = unit ? launch<T, V, TRI, true>(l, q) : launch<T, V, TRI, false>(l, q);
  else *handled = unit ? launch<T, 1, TRI, true>(l, q) : launch<T, 1, TRI, false>(l, q);
  return *handled ? check_launch() : B2_STATUS_OK;
}

}  // namespace ts
}  // namespace b2
