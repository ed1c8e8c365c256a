// Small and middle-sized gemv, symv and trmv (column sums) in one launch (Section 6.2.2): every output is gathered by one cluster.
//
// What bounds such a call is latency: launches, passes over partial sums, barriers.  A cluster of 1 .. 8 blocks
// owns 32 outputs and reads everything they depend on -- 32 rows of the canonical row-major view (row part), 32
// columns of it (column part), or, for symv, the 32 rows of the stored triangle up to the diagonal and the 32
// columns beyond it.  symv so reads each element twice, the second time from L2 where matrices of this size stay;
// in exchange no sum leaves the cluster: its blocks take the chunks of the contraction in turn and hand their 32
// sums to rank 0 through distributed shared memory, which writes y.  One launch, no workspace, no second pass.
//   row part:    a warp holds 4 rows, 64 packs of each in flight per chunk; rows are dealt to the warps modulo 8, so
//                that all rows of a warp start the same number of elements past a 16-byte boundary (8 lda is a
//                multiple of the pack length) and packs can be read aligned, the columns shifted by that number.
//   column part: a lane per column, so an instruction reads one 128-byte (256-byte) run of a row whatever its
//                alignment.  (Packs, several rows per instruction: a third slower at n = 3000 in double.)
//
// trmv overwrites x while other clusters still need it: every block first copies the part of x that it reads into
// shared memory and counts itself in the control block.  A cluster that finds all blocks counted writes its outputs;
// one that does not (a block has not even started) leaves them in the workspace under a flag, and the last block to
// be counted writes them at its end.  Nobody waits.
#pragma once

#include <algorithm>

#include "level2.cuh"

namespace b2 {
namespace ga {

constexpr int R = 32;             // outputs per cluster
constexpr int RPW = R / kWarps;   // rows of a warp in the row part
constexpr int kMaxGroups = 896;   // flags in the control block
constexpr int kMaxCluster = 8;
constexpr int CL = 16;            // loads of a thread in flight in the column part
constexpr int CB = CL * kWarps;   // rows of a batch there
constexpr int64_t kMaxBytesPerBlock = 128 * 1024;  // matrix bytes a block may be given: four chunks of latency

template <typename T>
struct Args {
  const T* a;
  int64_t lda;
  const T* x;  // base per vec_base()
  int64_t incx;
  T* y;
  int64_t incy;
  T alpha, beta;
  T* late;        // [groups * R] outputs that could not be written yet (in-place kinds)
  unsigned* ctl;  // counters, flags (in-place kinds)
  int defer;      // tests: take the late way first
  int rows, cols;
};

template <typename T>
__device__ __forceinline__ T ld_x(const T* p) { return B2_GUARD(p, sizeof(T)) ? *p : T(0); }

// ROWOUT / COLOUT of the kind: row part / column part.  Triangular kinds that are not symmetric work in place (and
// have a column part only: see run()).
template <typename T, bool AL, class K>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 8 ? 3 : 4) gather_kernel(const Args<T> p) {
  constexpr int V = VecLen<T>::value, SH = AL ? 0 : V - 1;
  constexpr int CH = 2 * 32 * V;                              // columns of a row-part chunk
  constexpr bool INPLACE = K::TRI != TRI_FULL && !K::SYM;
  static_assert(!(INPLACE && K::ROWOUT), "row sums are not formed in place");
  using P = Pack<T, V>;
  __shared__ T s_row[R], s_col[kWarps][R], s_sum[kMaxCluster][R];
  __shared__ int s_last;
  __shared__ unsigned s_mine[INPLACE ? kThreads : 1];
  extern __shared__ __align__(16) unsigned char gather_smem[];
  const int tid = (int)threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = (int)cluster_rank(), nr = (int)cluster_size();
  const int g = (int)blockIdx.x / nr, o0 = g * R;
  const unsigned long long a_el = (unsigned long long)p.a / sizeof(T);
  // columns of the row part, rows of the column part
  const int rlo = K::TRI == TRI_UPPER ? o0 : 0, rhi = K::TRI == TRI_LOWER ? min(p.cols, o0 + R) : p.cols;
  const int clo = K::TRI == TRI_LOWER ? o0 : 0, chi = K::TRI == TRI_UPPER ? min(p.rows, o0 + R) : p.rows;
  const int k0 = rlo / CH, nrow = K::ROWOUT ? (rhi + SH - 1) / CH + 1 - k0 : 0;
  const int nbat = K::COLOUT ? (chi - clo + CB - 1) / CB : 0;
  if (nr > 1) cluster_arrive();  // (completed below: every block of the cluster is running)
  grid_dep_wait();
  grid_dep_launch();

  const T* xp = p.x;
  int64_t xi = p.incx;
  bool last_reader = false;
  if (INPLACE) {
    T* xs = reinterpret_cast<T*>(gather_smem);
    const int lo = clo, hi = chi;
    for (int t0 = lo + tid; t0 < hi; t0 += 8 * kThreads) {  // eight loads in flight
      T v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = t0 + u * kThreads < hi ? ld_x(p.x + (int64_t)(t0 + u * kThreads) * p.incx) : T(0);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (t0 + u * kThreads < hi) xs[t0 + u * kThreads - lo] = v[u];
    }
    xp = xs - lo;
    xi = 1;
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      s_last = atomicAdd(p.ctl, 1u) == gridDim.x - 1;
    }
  }
  // (x of an in-place kind lies in shared memory, where the checking build's extents do not reach)
  auto x_at = [&](int j) { return INPLACE ? xp[j] : ld_x(xp + (int64_t)j * xi); };

  T rsum[RPW], csum = T(0);
#pragma unroll
  for (int u = 0; u < RPW; ++u) rsum[u] = T(0);

  if (K::ROWOUT) {
    const int s = AL ? 0 : (int)((a_el + (unsigned long long)warp * (unsigned long long)p.lda) % V);
    const T* const a0 = p.a + (int64_t)(o0 + warp) * p.lda + (lane * V - s);
    const int64_t rstride = (int64_t)kWarps * p.lda;
    const bool all_rows = o0 + R <= p.rows;
#pragma unroll 1
    for (int t = rank; t < nrow; t += nr) {
      const int c0 = (k0 + t) * CH;
      const bool fast = all_rows && c0 >= SH && c0 + CH <= p.cols &&
                        (K::TRI == TRI_FULL || (K::TRI == TRI_LOWER ? c0 + CH - 1 < o0 : c0 - SH > o0 + R - 1));
      P av[RPW][2];
      T xv[2][V];
      if (fast) {
#pragma unroll
        for (int u = 0; u < RPW; ++u)
#pragma unroll
          for (int h = 0; h < 2; ++h) av[u][h] = ld_nc<T, V>(a0 + u * rstride + c0 + h * 32 * V);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int e = 0; e < V; ++e) xv[h][e] = x_at(c0 + h * 32 * V + lane * V - s + e);
#pragma unroll
        for (int u = 0; u < RPW; ++u)
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int e = 0; e < V; ++e) rsum[u] = av[u][h].v[e] * xv[h][e] + rsum[u];
      } else {
        // packs that exist go out together, each under its predicate; those the matrix edge cuts element by element
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int c = c0 + h * 32 * V + lane * V - s;
          const bool whole = c >= 0 && c + V <= p.cols;
#pragma unroll
          for (int u = 0; u < RPW; ++u) {
            const int i = o0 + u * kWarps + warp;
            const bool in = i < p.rows && (K::TRI == TRI_FULL || (K::TRI == TRI_LOWER ? c <= i : c + V - 1 >= i));
            av[u][h] = ld_nc_if<T, V>(a0 + u * rstride + c0 + h * 32 * V, whole && in);
          }
#pragma unroll
          for (int e = 0; e < V; ++e) {
            const bool in = c + e >= rlo && c + e < rhi;
            xv[h][e] = ld_el_if<T>(xp + (int64_t)(c + e) * xi, in);
          }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int c = c0 + h * 32 * V + lane * V - s;
          if (!(c >= 0 && c + V <= p.cols) && c + V > 0 && c < p.cols) {
#pragma unroll
            for (int u = 0; u < RPW; ++u)
#pragma unroll
              for (int e = 0; e < V; ++e)
                av[u][h].v[e] = ld_el_if<T>(a0 + u * rstride + c0 + h * 32 * V + e, o0 + u * kWarps + warp < p.rows && c + e >= 0 && c + e < p.cols);
          }
#pragma unroll
          for (int u = 0; u < RPW; ++u) {
            const int i = o0 + u * kWarps + warp;
#pragma unroll
            for (int e = 0; e < V; ++e) {
              const int j = c + e;
              bool in = i < p.rows && j >= 0 && j < p.cols;
              if (K::TRI == TRI_LOWER) in = in && j <= i;
              if (K::TRI == TRI_UPPER) in = in && j >= i;
              const T v = (K::UNIT && j == i) ? T(1) : av[u][h].v[e];
              rsum[u] = in ? v * xv[h][e] + rsum[u] : rsum[u];  // (a select: what is not referenced may be anything)
            }
          }
        }
      }
    }
    const T v = multi_group_sum<32, RPW>(rsum, lane);
    constexpr int LPV = 32 / RPW;
    if (lane % LPV == 0) s_row[lane / LPV * kWarps + warp] = v;
  }
  if (K::COLOUT) {
    const int j = o0 + lane;
    const bool all_cols = o0 + R <= p.cols;
    const int64_t rstride = (int64_t)kWarps * p.lda;
    int t = rank - nrow % nr;  // (the row part's chunks come first in the blocks' turns)
    if (t < 0) t += nr;
#pragma unroll 1
    for (; t < nbat; t += nr) {
      const int r0 = clo + t * CB;
      const bool fast = all_cols && r0 + CB <= chi && (K::TRI == TRI_FULL || (K::TRI == TRI_LOWER ? r0 > o0 + R - 1 : r0 + CB - 1 < o0));
      T av[CL], xv[CL];
      const T* at = p.a + (int64_t)(r0 + warp) * p.lda + j;
      if (fast) {
#pragma unroll
        for (int u = 0; u < CL; ++u) av[u] = __ldg(at + u * rstride);
#pragma unroll
        for (int u = 0; u < CL; ++u) xv[u] = x_at(r0 + warp + u * kWarps);
#pragma unroll
        for (int u = 0; u < CL; ++u) csum = av[u] * xv[u] + csum;
      } else {
#pragma unroll
        for (int u = 0; u < CL; ++u) {
          const int i = r0 + warp + u * kWarps;
          bool in = i < chi && j < p.cols;
          if (K::TRI == TRI_LOWER) in = in && (K::SYM ? j < i : j <= i);
          if (K::TRI == TRI_UPPER) in = in && (K::SYM ? j > i : j >= i);
          av[u] = ld_el_if<T>(at + u * rstride, in && !(K::UNIT && j == i));
          if (K::UNIT && in && j == i) av[u] = T(1);
          // (zero where the element is masked: x may hold infinities where the triangle ends)
          if constexpr (INPLACE) xv[u] = in ? x_at(i) : T(0);
          else xv[u] = ld_el_if<T>(xp + (int64_t)i * xi, in);
        }
#pragma unroll
        for (int u = 0; u < CL; ++u) csum = av[u] * xv[u] + csum;
      }
    }
    s_col[warp][lane] = csum;
  }
  __syncthreads();
  if (INPLACE) last_reader = s_last != 0;
  if (nr > 1) cluster_wait();
  if (warp == 0) {
    T v = K::ROWOUT ? s_row[lane] : T(0);
    if (K::COLOUT) {
#pragma unroll
      for (int w = 0; w < kWarps; ++w) v += s_col[w][lane];
    }
    if (rank == 0) s_sum[0][lane] = v;
    else st_rank0(&s_sum[rank][lane], v);
  }
  if (nr > 1) {
    cluster_arrive();
    cluster_wait();
  }
  const int nout = K::ROWOUT ? p.rows : p.cols;
  auto write = [&](int i, T v) {
    T* yp = p.y + (int64_t)i * p.incy;
    B2_STORE(yp, p.beta != T(0) ? p.alpha * v + p.beta * *yp : p.alpha * v);
  };
  if (rank == 0 && warp == 0) {
    T v = s_sum[0][lane];
    for (int c = 1; c < nr; ++c) v += s_sum[c][lane];
    if (!INPLACE) {
      if (o0 + lane < nout) write(o0 + lane, v);
    } else {
      volatile unsigned* const readers = p.ctl;
      unsigned* const flag = p.ctl + 2 + g;
      bool now = false;
      if (lane == 0) now = !p.defer && *readers == gridDim.x;
      now = __shfl_sync(0xffffffffu, (int)now, 0) != 0;
      if (!now) {  // some block has not read its x yet
        p.late[o0 + lane] = v;
        __threadfence();
        __syncwarp();
        if (lane == 0) {
          atomicExch(flag, 1u);
          __threadfence();
          if (*readers == gridDim.x) now = atomicCAS(flag, 1u, 0u) == 1u;  // all have by now: nobody may come for it
        }
        now = __shfl_sync(0xffffffffu, (int)now, 0) != 0;
      }
      if (now) {
        __threadfence();
        if (o0 + lane < nout) write(o0 + lane, v);
      }
    }
  }
  if (INPLACE) {
    if (last_reader) {  // outputs left behind before this block had read its x
      const int ngroups = (int)gridDim.x / nr;
      __threadfence();
      for (int q0 = 0; q0 < ngroups; q0 += kThreads) {
        if (q0 + tid < ngroups) s_mine[tid] = atomicCAS(p.ctl + 2 + q0 + tid, 1u, 0u);
        __syncthreads();
        __threadfence();
        const int n = min(kThreads, ngroups - q0) * R;
#pragma unroll 4
        for (int t = tid; t < n; t += kThreads) {
          const int i = q0 * R + t;
          if (s_mine[t / R] == 1u && i < nout) write(i, __ldcg(p.late + i));
        }
        __syncthreads();
      }
    }
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      if (atomicAdd(p.ctl + 1, 1u) == gridDim.x - 1) p.ctl[0] = p.ctl[1] = 0u;  // the last block leaves the counters clean
    }
  }
}

// Launches the kernel; *handled is false (nothing launched) where the sizes do not allow it.
template <typename T, bool AL, class K>
static int launch(const Launch& l, const L2Args<T>& q, bool* handled, bool one_launch) {
  constexpr int V = VecLen<T>::value, CH = 2 * 32 * V;
  constexpr bool INPLACE = K::TRI != TRI_FULL && !K::SYM;
  const int64_t nout = K::ROWOUT ? q.rows : q.cols, len = K::ROWOUT ? q.cols : q.rows;
  const int64_t groups = (nout + R - 1) / R;
  if (groups > kMaxGroups || len > (1 << 24)) return B2_STATUS_OK;
  const size_t smem = INPLACE ? (size_t)len * sizeof(T) : 0;
  if (smem > 40 * 1024 || (INPLACE && (size_t)groups * R * sizeof(T) > l.scratch_bytes)) return B2_STATUS_OK;
  // blocks per cluster: no more than there are chunks, and one resident wave in all
  const int64_t items = (K::ROWOUT ? (len + CH - 1) / CH : 0) + (K::COLOUT ? (len + CB - 1) / CB : 0);
  const int64_t wave = (int64_t)sm_count() * (sizeof(T) == 8 ? 3 : 4);
  int nr = 1;
  while (nr < kMaxCluster && 2 * nr <= items && groups * nr * (INPLACE ? 2 : 1) <= wave) nr *= 2;
  const int64_t bytes = q.rows * q.cols * (int64_t)sizeof(T) / (INPLACE ? 2 : 1);
  if (knob(kKnobGather) < 2) {  // (see run())
    if (bytes > kMaxBytesPerBlock * groups * nr) return B2_STATUS_OK;
    const bool turns = items > nr, late = groups * nr * 8 > wave * 7;
    if (K::TRI == TRI_FULL && K::ROWOUT &&
        ((late && !(sizeof(T) == 8 && items == 1)) || (turns && nr <= 2) ||
         (one_launch && (turns || (!AL && len <= (sizeof(T) == 4 ? 768 : 512)))))) return B2_STATUS_OK;
    if (K::TRI == TRI_FULL && K::COLOUT && sizeof(T) == 4 && AL && (late || items > 4 * nr)) return B2_STATUS_OK;
  }
  Args<T> p = {};
  p.a = q.a;
  p.lda = q.lda;
  p.x = K::ROWOUT ? q.xc : q.xr;
  p.incx = K::ROWOUT ? q.incxc : q.incxr;
  p.y = q.y;
  p.incy = q.incy;
  p.alpha = q.alpha;
  p.beta = q.beta;
  p.late = reinterpret_cast<T*>(l.scratch);
  p.ctl = l.ctl + kCtlGather;
  p.defer = knob(kKnobGather) == 3;
  p.rows = (int)q.rows;
  p.cols = (int)q.cols;
  *handled = true;
  launch_clusters(gather_kernel<T, AL, K>, (unsigned)(groups * nr), (unsigned)nr, dim3(kThreads), smem, l.stream, p);
  return check_launch();
}
// Where one launch by clusters is the faster way: up to a matrix size (of the whole square, where a triangle is read).
// Against the tile kernels and their second pass, three matrices in turn, tile kernel / this one in us (each product
// repeated; "both": the two products of a pass one after the other, which read the matrix through different SMs), with
// the last size where this one wins and the first where it does not:
//   gemv row part   the blocks must fit one wave: a second one costs more than the second pass (double 4000 x 400, 12.8
//                   MB, 4.1 / 5.6), except in double where a row is a single chunk (16000 x 128 5.1 / 3.7).  Where the
//                   tile kernel needs no second pass either (one_launch: short rows) it is the faster one as soon as
//                   blocks here take turns (float 4899 x 612, 12 MB, 4.5 / 6.1; 8 MB 4.7 / 3.7), and off 16-byte
//                   boundaries nearly always (double 2000 x 256 2.7 / 3.9, float 4000 x 512 4.0 / 4.9, 1000 x 707
//                   3.8 / 4.5, but 1000 x 1000 4.5 / 3.5).  Float 16 MB 5.2 / 4.8, 24 6.4 / 5.8, 32 7.4 / 7.6 (866 x 6928
//                   and like it); double 50 11.7 / 11.2, 64 13.4 / 13.5; unaligned to 100 MB and beyond (21.2 / 18.5).
//   gemv column part  float 16 MB 6.3 / 5.8, 20 7.0 / 7.4, one wave of blocks here too (707 x 5656 6.2 / 7.8) and no more
//                   than four turns of them (both, 4896 x 608, 10.2 / 10.8 to 13.8); double 20 8.2 / 6.6, 24 7.4 / 7.5
//                   (32 11.7 / 9.2, but 36 9.6 / 11.6); unaligned float 32 12.6 / 12.5, 40 13.6 / 15.1, double 64
//                   16.7 / 15.5, 80 18.6 / 22.3.
//   trmv row part   never, and not built: the tile kernel's second pass costs less than the in-place protocol (n = 64
//                   4.6 / 4.9, 512 4.6 / 5.7, 3008 in float 6.9 / 9.2; unaligned 4.6 / 4.9, 5.9 / 6.2, n = 3001 8.7 / 10.5).
//   trmv column part  both, lower and upper triangle: float 4 MB 12.8 / 10.9 and 12.1 / 11.9, 6 MB 12.6 / 11.3 and
//                   12.2 / 13.3; double 18 13.3 / 13.2 and 13.8 / 14.2, 20 13.1 / 16.0 and 13.8 / 13.7 (equal from 32 to 50);
//                   unaligned float 49 MB 22.6 / 22.1, 58 23.2 / 25.5, 74 25.7 / 28.9 (with a copy and the row product), double the
//                   same on twelve matrices, four views, 5 MB 11.8 - 12.0 / 11.8 - 12.9, 7.2 12.1 - 12.4 / 12.8 - 13.6, 9.7 14.0 - 15.2 /
//                   14.3 - 15.0, 32 17.1 - 17.9 / 17.9 - 19.4, 98 25.5 - 27.3 / 28.2 - 30.6 (on three 5.8 12.8 / 11.9 - 12.6, 8 equal).
//   symv            reads its elements twice: float (ring kernel, both triangles) n = 1520 14.2 / 12.6, 1664 12.2 / 12.8, 2048 12.4 /
//                   13.7, 2100 15.3 / 14.8, 2176 13.6 / 14.5, with room for its partials; double 20 MB
//                   7.6 / 6.5, 24 7.5 / 7.6; unaligned (both triangles) float 21 MB 20.5 / 19.3, 23 20.5 / 20.5, 29 21.4 / 23.5, 35
//                   23.0 / 26.6, double 29 22.8 / 19.0, 32 23.1 / 23.0, 35 23.8 / 24.8, 72 32.3 / 35.0.
// room: whether the tile kernels' partials fit the workspace without much longer blocks; where they do not, this kernel, which
// needs none or one vector, goes on off 16-byte boundaries (64 KB of scratch, us, tile kernel / this one: trmv in float n = 3001 32.9 / 13.2,
// 4001 58.8 / 15.6, double 3001 75.0 / 13.0; symv in float n = 2501 with 264 KB 20.6 / 10.5, 3501 with 464 38.5 / 15.7, with less none).
template <typename T, class K>
constexpr int64_t max_mb(bool al, bool room) {
  constexpr bool F = sizeof(T) == 4;
  if (!al && !room && K::SYM) return F ? 85 : 80;
  if (!al && !room && K::TRI != TRI_FULL) return F ? 85 : 101;
  if (K::SYM) return al ? (F ? (room ? 11 : 20) : 22) : (F ? 23 : 33);
  if (K::TRI != TRI_FULL) return al ? (F ? 5 : 18) : (F ? 50 : 7);
  if (K::ROWOUT) return al ? (F ? 24 : 50) : 110;
  return al ? (F ? 17 : 22) : (F ? 35 : 70);
}
template <typename T, class K>
static int run(const Launch& l, const L2Args<T>& q, bool* handled, bool one_launch = false, bool room = true) {
  *handled = false;
  if (knob(kKnobGather) == 0) return B2_STATUS_OK;
  const bool al = aligned_to(q.a, 16) && q.lda % VecLen<T>::value == 0;
  if (knob(kKnobGather) < 2 && (double)q.rows * (double)q.cols * sizeof(T) > (double)max_mb<T, K>(al, room) * 1e6) return B2_STATUS_OK;
  return al ? launch<T, true, K>(l, q, handled, one_launch) : launch<T, false, K>(l, q, handled, one_launch);
}

}  // namespace ga
}  // namespace b2
