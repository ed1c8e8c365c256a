// ger: A <- alpha*x*y^T + A (Section 6.2.2; the paper's Figure 7 caption notes that ger shares
// the gemv schedule).  Pure streaming read-modify-write of A: each lane keeps alpha*y_j for
// its columns in registers and reuses them down a band of rows, x_i is a broadcast load.
#include "level2.cuh"
#include "skinny.cuh"

namespace b2 {

// Blocks per SM at least (0: as the compiler likes it): the tiles of a cut matrix, with all their loads in flight, would
// otherwise take the registers of one of two blocks (packs: 509117 x 32 in double 41 us, 54 with one block) or of one
// of four (double elements: 100003 x 64 18.8 and 20.4 us; in float the bound only makes the compiler use more).
template <typename T, int V, class S>
constexpr int kGerBlocks = V > 1 ? 2 : sizeof(T) == 8 && S::CU == 1 ? 4 : 0;

// CUT: the kernel knows rows that end inside a pack.  Short row segments (CU == 1) leave that to a kernel of its own: with
// the loads of cut packs in it the one for whole packs needs 141 registers instead of 92 in double, and bounded to 128 it
// lost 2 % (200 x 90000 by columns: 51.2 us without them, 52.4 with, 50.5 so).  Long ones have it all in one: the kernel for whole
// packs takes fewer registers than two resident blocks leave it, and a third one costs 2-5 % (4096 x 4096 in float
// 23.1 -> 23.6 us, 6000 x 3000 25.3 -> 26.7).
template <typename T, int V, class S, bool CUT>
__global__ void __launch_bounds__(kThreads, kGerBlocks<T, V, S>) ger_kernel(T* __restrict__ a, int64_t lda, int64_t rows, int64_t cols,
                                                       const T* __restrict__ xr, int64_t incxr,
                                                       const T* __restrict__ yc, int64_t incyc, T alpha,
                                                       int64_t rows_per_cta, int nct) {
  grid_dep_wait();
  grid_dep_launch();
  constexpr int LPR = S::LPR, CU = S::CU, RU = S::RU, G = S::G, RB = S::RB;
  constexpr int TC = LPR * V * CU;
  using P = Pack<T, V>;
  // Packs, and single elements of which a warp takes 128 in a row: the sectors are written whole, or nearly so, and the
  // matrix passes through L2 evict-first, loads and stores.  Elements of short rows leave partly written sectors: loaded
  // evict-first they were gone from L2 when the stores came, and had to be filled again (1000000 x 16, lda 19, in
  // double 80 us, 48 so); those of cut tiles are stored plainly (streaming, 100003 x 64 in float 9.9 -> 10.2 us).  Long
  // rows off 16-byte boundaries, float, with plain L2 loads -> evict-first -> streaming stores of cut tiles too: 16000 x
  // 8000 178.2 -> 170.5 -> 167.9 us, 5001 x 5000 37.2 -> 36.2 -> 36.2, 100000 x 300 45.8 -> 44.6 -> 42.7; double 309 ->
  // 308 -> 305, 62.1 -> 62.0 -> 62.1, 77.2 -> 77.6 -> 73.5; streaming stores of whole tiles against plain ones
  // 37.2 / 37.7 (5001 x 5000, float), 26.8 / 27.4 (509117 x 32), 94.1 / 87.0 (500000 x 100).
  constexpr bool EVICT = V > 1 || CU > 1;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane / LPR, q = lane % LPR;
  const int ct = blockIdx.x % nct;
  const int64_t rs = blockIdx.x / nct;
  const int64_t r_begin = rs * rows_per_cta, r_end = min(rows, r_begin + rows_per_cta);
  const int64_t c0 = (int64_t)ct * TC;
  T yv[CU][V];
#pragma unroll
  for (int u = 0; u < CU; ++u)
#pragma unroll
    for (int e = 0; e < V; ++e) {
      const int64_t j = c0 + (u * LPR + q) * V + e;
      yv[u][e] = j < cols ? alpha * __ldg(yc + j * incyc) : T(0);
    }
  for (int64_t rb = r_begin; rb < r_end; rb += RB) {
    int64_t rowi[RU];
    T xv[RU];
#pragma unroll
    for (int ru = 0; ru < RU; ++ru) {
      rowi[ru] = rb + (ru * kWarps + warp) * G + g;
      xv[ru] = rowi[ru] < r_end ? __ldg(xr + rowi[ru] * incxr) : T(0);
    }
    if (rb + RB <= r_end && c0 + TC <= cols) {
      P av[RU][CU];
#pragma unroll
      for (int ru = 0; ru < RU; ++ru)
#pragma unroll
        for (int u = 0; u < CU; ++u) {
          const T* ap = a + rowi[ru] * lda + c0 + (u * LPR + q) * V;
          av[ru][u] = EVICT ? ld_cs<T, V>(ap) : ld_cg<T, V>(ap);
        }
#pragma unroll
      for (int ru = 0; ru < RU; ++ru)
#pragma unroll
        for (int u = 0; u < CU; ++u) {
#pragma unroll
          for (int e = 0; e < V; ++e) av[ru][u].v[e] = xv[ru] * yv[u][e] + av[ru][u].v[e];
          st_cs<T, V>(a + rowi[ru] * lda + c0 + (u * LPR + q) * V, av[ru][u]);
        }
    } else if (V > 1 && (!CUT || c0 + TC <= cols || (cols - c0) % V == 0)) {
      // only the matrix edge cuts this tile, on pack boundaries (narrow matrices, short row
      // bands): the loads still go out together, each under its own row / pack predicate.
      const int64_t npk = (min(cols, c0 + TC) - c0) / V;  // packs of this tile that exist
      P av[RU][CU];
#pragma unroll
      for (int ru = 0; ru < RU; ++ru)
#pragma unroll
        for (int u = 0; u < CU; ++u) {
          const T* ap = a + rowi[ru] * lda + c0 + (u * LPR + q) * V;
          const bool in = rowi[ru] < r_end && u * LPR + q < npk;
          if constexpr (CU == 1) av[ru][u] = ld_cg_if<T, V>(ap, in);
          else if (in) av[ru][u] = ld_cs<T, V>(ap);  // (as one predicated instruction: the registers again)
        }
#pragma unroll
      for (int ru = 0; ru < RU; ++ru)
#pragma unroll
        for (int u = 0; u < CU; ++u)
          if (rowi[ru] < r_end && u * LPR + q < npk) {
#pragma unroll
            for (int e = 0; e < V; ++e) av[ru][u].v[e] = xv[ru] * yv[u][e] + av[ru][u].v[e];
            st_cs<T, V>(a + rowi[ru] * lda + c0 + (u * LPR + q) * V, av[ru][u]);
          }
    } else if constexpr (V == 1 || CUT) {
      // rows that end inside a pack, element-wise tiles: the loads go out together all the same
      P av[RU][CU];
#pragma unroll
      for (int ru = 0; ru < RU; ++ru)
#pragma unroll
        for (int u = 0; u < CU; ++u) {
          const int64_t cv = c0 + (u * LPR + q) * V;
          T* ap = a + rowi[ru] * lda + cv;
          av[ru][u] = ld_cg_if<T, V>(ap, rowi[ru] < r_end && cv + V <= cols);
          if (V > 1 && cv < cols && cv + V > cols) {
#pragma unroll
            for (int e = 0; e < V; ++e) av[ru][u].v[e] = ld_cg_if<T, 1>(ap + e, rowi[ru] < r_end && cv + e < cols).v[0];
          }
        }
#pragma unroll
      for (int ru = 0; ru < RU; ++ru)
#pragma unroll
        for (int u = 0; u < CU; ++u) {
          const int64_t cv = c0 + (u * LPR + q) * V;
          T* ap = a + rowi[ru] * lda + cv;
          if (rowi[ru] >= r_end) continue;
#pragma unroll
          for (int e = 0; e < V; ++e) av[ru][u].v[e] = xv[ru] * yv[u][e] + av[ru][u].v[e];
          if (V > 1 && cv + V <= cols) {
            st_cs<T, V>(ap, av[ru][u]);
          } else {
#pragma unroll
            for (int e = 0; e < V; ++e)
              if (cv + e < cols) {
                if constexpr (V == 1 && EVICT) st_cs<T, 1>(ap, av[ru][u]);
                else B2_STORE(ap + e, av[ru][u].v[e]);
              }
          }
        }
    }
  }
}

// Unpadded matrices whose rows start off 16-byte boundaries (odd widths): the matrix is one contiguous run, so its
// packs are aligned even though its rows are not.  A thread divides once per chunk for the row and column of its first
// pack, the others are a fixed number of rows and columns further on; y comes through L1, x is nearly a broadcast.
// (The element-wise tiles: 1000001 x 31 float 120 us, 4097 x 4095 28 us; a third and three quarters of the rate.)
constexpr int kFlatPacks = 4;
template <typename T>
__global__ void __launch_bounds__(kThreads) flat_ger_kernel(T* __restrict__ a, unsigned total, unsigned head, unsigned nvec, unsigned cols,
                                                            const T* __restrict__ xr, int64_t incxr, const T* __restrict__ yc, int64_t incyc,
                                                            T alpha, unsigned step_rows, unsigned step_cols) {
  grid_dep_wait();
  grid_dep_launch();
  constexpr int V = VecLen<T>::value, NV = kFlatPacks;
  using P = Pack<T, V>;
  const unsigned v0 = blockIdx.x * (unsigned)(kThreads * NV) + threadIdx.x;
  P av[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const unsigned v = v0 + k * kThreads;
    av[k] = ld_cg_if<T, V>(a + head + (size_t)v * V, v < nvec);
  }
  unsigned e0 = head + v0 * V, row = e0 / cols, col = e0 - row * cols;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const unsigned v = v0 + k * kThreads;
    if (v < nvec) {
      unsigned i = row, j = col;
      T xi = alpha * __ldg(xr + (int64_t)i * incxr);
#pragma unroll
      for (int e = 0; e < V; ++e) {
        av[k].v[e] = xi * __ldg(yc + (int64_t)j * incyc) + av[k].v[e];
        if (++j == cols && e + 1 < V) {
          j = 0;
          xi = alpha * __ldg(xr + (int64_t)++i * incxr);
        }
      }
      st_cs<T, V>(a + head + (size_t)v * V, av[k]);
    }
    row += step_rows, col += step_cols;
    if (col >= cols) col -= cols, ++row;
  }
  if (blockIdx.x == 0) {  // the elements before the first and after the last pack
    const unsigned tail0 = head + nvec * V, n = head + (total - tail0);
    if (threadIdx.x < n) {
      const unsigned t = threadIdx.x < head ? threadIdx.x : tail0 + (threadIdx.x - head), i = t / cols, j = t - i * cols;
      T* ap = a + t;
      B2_STORE(ap, alpha * __ldg(xr + (int64_t)i * incxr) * __ldg(yc + (int64_t)j * incyc) + *ap);
    }
  }
}

template <typename T>
static int flat_ger(const Launch& l, T* a, int64_t rows, int64_t cols, const T* xr, int64_t incxr, const T* yc, int64_t incyc, T alpha) {
  constexpr int V = VecLen<T>::value;
  const unsigned total = (unsigned)(rows * cols);
  unsigned head = (unsigned)((16 - reinterpret_cast<uintptr_t>(a) % 16) % 16 / sizeof(T));
  if (head > total) head = total;
  const unsigned nvec = (total - head) / V, per = kThreads * kFlatPacks, step = kThreads * V;
  launch_chained(flat_ger_kernel<T>, dim3(nvec ? (nvec + per - 1) / per : 1), dim3(kThreads), 0, l.stream, a, total, head, nvec, (unsigned)cols, xr,
                 incxr, yc, incyc, alpha, step / (unsigned)cols, step % (unsigned)cols);
  return check_launch();
}

template <typename T, int V, class S>
static int ger_launch(const Launch& l, T* a, int64_t lda, int64_t rows, int64_t cols, const T* xr, int64_t incxr,
                      const T* yc, int64_t incyc, T alpha) {
  constexpr int TC = S::template tc<V>();
  const int nct = (int)((cols + TC - 1) / TC);
  const int64_t rows_per_cta = (int64_t)S::RB * knob(kKnobGerRows);
  const int64_t nrs = (rows + rows_per_cta - 1) / rows_per_cta;
  if (nrs * nct > 0x7fffffff) return B2_STATUS_NOT_IMPLEMENTED;
  auto kern = ger_kernel<T, V, S, (V > 1)>;
  if constexpr (V > 1 && S::CU == 1)
    if (cols % V == 0) kern = ger_kernel<T, V, S, false>;
  launch_chained(kern, dim3((unsigned)(nrs * nct)), dim3(kThreads), 0, l.stream, a, lda, rows, cols, xr, incxr, yc, incyc, alpha,
                 rows_per_cta, nct);
  return check_launch();
}

template <typename T, int V>
static int ger_shape(const Launch& l, T* a, int64_t lda, int64_t rows, int64_t cols, const T* xr, int64_t incxr,
                     const T* yc, int64_t incyc, T alpha) {
  const int64_t nv = (cols + V - 1) / V;
  if (nv >= 128) return ger_launch<T, V, ShapeWide>(l, a, lda, rows, cols, xr, incxr, yc, incyc, alpha);
  if (nv > 16) return ger_launch<T, V, ShapeMid>(l, a, lda, rows, cols, xr, incxr, yc, incyc, alpha);
  if (nv > 8) return ger_launch<T, V, ShapeHalf>(l, a, lda, rows, cols, xr, incxr, yc, incyc, alpha);
  return ger_launch<T, V, ShapeQuarter>(l, a, lda, rows, cols, xr, incxr, yc, incyc, alpha);
}

template <typename T>
static int ger_impl(const b2_ctx* ctx, int order, int64_t m, int64_t n, T alpha, const T* x, int64_t incx, const T* y,
                    int64_t incy, T* a, int64_t lda) {
  if (order != B2_ROW_MAJOR && order != B2_COL_MAJOR) return -1;
  if (m < 0) return -2;
  if (n < 0) return -3;
  if (incx == 0) return -6;
  if (m > 0 && n > 0 && (x == nullptr || !aligned_to(x, sizeof(T)))) return -5;
  if (incy == 0) return -8;
  if (m > 0 && n > 0 && (y == nullptr || !aligned_to(y, sizeof(T)))) return -7;
  if (m > 0 && n > 0 && (a == nullptr || !aligned_to(a, sizeof(T)))) return -9;
  const int64_t minor = order == B2_ROW_MAJOR ? n : m;
  if (lda < (minor > 1 ? minor : 1)) return -10;
  Launch l;
  if (int st = make_launch(ctx, &l)) return st;
  if (m == 0 || n == 0 || alpha == T(0)) return B2_STATUS_OK;
  B2_DBG_RANGE(l, a, (size_t)(((order == B2_ROW_MAJOR ? m : n) - 1) * lda + minor) * sizeof(T));
  B2_DBG_VEC(l, x, m, incx);
  B2_DBG_VEC(l, y, n, incy);
  B2_DBG_COMMIT(l);
  // canonical row-major view: row vector index = slow dimension of the buffer
  const bool rm = order == B2_ROW_MAJOR;
  const int64_t rows = rm ? m : n, cols = rm ? n : m;
  const T* xr = rm ? vec_base(x, m, incx) : vec_base(y, n, incy);
  const int64_t incxr = rm ? incx : incy;
  const T* yc = rm ? vec_base(y, n, incy) : vec_base(x, m, incx);
  const int64_t incyc = rm ? incy : incx;
  constexpr int V = VecLen<T>::value;
  // (measured: the element-wise walk wins in double; in float the pack kernels stay ahead)
  if (knob(kKnobNarrowBlock) && sizeof(T) == 8 && wide_applies<T>(rows, cols)) {
    const int64_t want = (cols + kThreads - 1) / kThreads, cap = (int64_t)sm_count() * 8;
    launch_chained(wide_ger_kernel<T>, dim3((unsigned)(want < cap ? want : cap)), dim3(kThreads), 0, l.stream, a, lda, (int)rows, cols, xr, incxr, yc, incyc,
                                                                                alpha);
    return check_launch();
  }
  if (skinny_applies(a, lda, rows, cols, false)) return skinny_ger<T>(l, a, rows, cols, xr, incxr, yc, incyc, alpha);
  if (aligned_to(a, 16) && lda % V == 0) return ger_shape<T, V>(l, a, lda, rows, cols, xr, incxr, yc, incyc, alpha);
  if (lda == cols && rows * (double)cols < 2147483648.0) return flat_ger<T>(l, a, rows, cols, xr, incxr, yc, incyc, alpha);
  return ger_shape<T, 1>(l, a, lda, rows, cols, xr, incxr, yc, incyc, alpha);
}

}  // namespace b2

extern "C" {
int b2_sger(const b2_ctx* ctx, int order, int64_t m, int64_t n, float alpha, const float* x, int64_t incx,
            const float* y, int64_t incy, float* a, int64_t lda) {
  return b2::ger_impl<float>(ctx, order, m, n, alpha, x, incx, y, incy, a, lda);
}
int b2_dger(const b2_ctx* ctx, int order, int64_t m, int64_t n, double alpha, const double* x, int64_t incx,
            const double* y, int64_t incy, double* a, int64_t lda) {
  return b2::ger_impl<double>(ctx, order, m, n, alpha, x, incx, y, incy, a, lda);
}
}
