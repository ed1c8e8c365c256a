// symv and trmv entry-point bodies (Section 6.2.2, "Triangular Matrix"): both run on the
// level-2 tile kernel restricted to one triangle of the canonical row-major view.
//   symv : row sums over the stored triangle (with the diagonal) plus column sums over its
//          strictly off-diagonal part -- each stored element is loaded once and used twice.
//   trmv : row sums (op(A) rows contiguous) or column sums (op(A) rows strided), the
//          diagonal replaced by 1 for diag = unit.  The result goes to partials first and is
//          written over x by the finalize kernel, after every block has finished reading x.
#pragma once
#include "level2.cuh"
#include "gather.cuh"
#include "tri_tile.cuh"
#include "trmv_small.cuh"

namespace b2 {

template <typename T>
static int check_square(int order, int64_t n, const T* a, int64_t lda, int arg_order, int arg_n, int arg_a,
                        int arg_lda) {
  if (order != B2_ROW_MAJOR && order != B2_COL_MAJOR) return -arg_order;
  if (n < 0) return -arg_n;
  if (n > 0 && (a == nullptr || !aligned_to(a, sizeof(T)))) return -arg_a;
  if (lda < (n > 1 ? n : 1)) return -arg_lda;
  return 0;
}

// Rows per block of the kinds with column sums: 3 1/4 blocks for each SM (480) that hold any of the triangle, as long as they
// keep 64 rows; longer blocks where the matrix is larger, up to what measured fastest (a block is a sequence of
// steps; off 16-byte boundaries, where a step takes longer, the last blocks are waited for longer).  Us, with 512 rows for
// all / with this rule: symv in float n = 4944 32.3 / 29.6, 4945 51.5 / 35.7, 6001 57.9 / 43.8, 9934 by columns 94 / 84, in double
// 3473 39.7 / 32.4; a copy and both products of trmv in double n = 3581 33.4 / 27.2, 3580 27.5 / 25.7, 11001 163 / 158; the same
// from n = 8000 on in float on aligned matrices (symv n = 8192 with 512, 256, 128 rows: 54.8, 55.4, 56.5).
template <typename T>
static int64_t tri_rows(const L2Args<T>& a, int tile_cols) {
  if (const int64_t k = knob(kKnobTriRows)) return k;
  const bool aligned = aligned_to(a.a, 16) && a.lda % VecLen<T>::value == 0;
  const int64_t most = !aligned ? 256 : sizeof(T) == 4 ? 512 : 384;
  const double rows = (double)a.rows * (double)a.cols / (2.0 * tile_cols * 3.25 * sm_count());
  return rows > (double)most ? most : std::min(most, std::max<int64_t>(64, (int64_t)(rows + 32) / 64 * 64));
}

template <typename T>
static L2Plan plan_tri(const L2Args<T>& a) {
  const int V = (aligned_to(a.a, 16) && a.lda % VecLen<T>::value == 0) || l2_shift(a, true, 0) ? VecLen<T>::value : 1;
  const int64_t nv = (a.cols + V - 1) / V;
  L2Plan p;
  p.shape = (nv >= 512 && !l2_shift(a, true, 0) && knob(kKnobTriWide)) ? SHAPE_WIDE : SHAPE_MID;
  p.ctiles_per_cta = 1;
  p.tile_cols = shape_packs_per_row(p.shape) * V;
  p.rows_per_cta = tri_rows(a, p.tile_cols);
  return p;
}

// Whether the workspace holds the partials of a kind with column sums (sym: row sums too) in blocks of up to twice the planned
// rows.  (With 800 KB symv in float n = 3501 takes 13.7 us so, 15.7 in the gather kernel; twice as long again 17.8 / 17.8 at 4001.)
template <typename T>
static bool tri_room(const Launch& l, const L2Args<T>& a, const L2Plan& p, bool sym) {
  const int64_t tiles = (a.cols + p.tile_cols - 1) / p.tile_cols, bands = (a.rows + 2 * p.rows_per_cta - 1) / (2 * p.rows_per_cta);
  const int64_t spill = l2_shift(a, sym, 0) ? bands * (tiles + 1) * (VecLen<T>::value - 1) : 0;
  return (size_t)(((sym ? tiles : 0) + bands) * a.cols + spill) * sizeof(T) + 512 <= l.scratch_bytes;
}

template <typename T>
static int symv_impl(const b2_ctx* ctx, int order, int uplo, int64_t n, T alpha, const T* a, int64_t lda, const T* x,
                     int64_t incx, T beta, T* y, int64_t incy) {
  if (int e = check_square(order, n, a, lda, 1, 3, 5, 6)) return e;
  if (uplo != B2_UPPER && uplo != B2_LOWER) return -2;
  if (incx == 0) return -8;
  if (n > 0 && (x == nullptr || !aligned_to(x, sizeof(T)))) return -7;
  if (incy == 0) return -11;
  if (n > 0 && (y == nullptr || !aligned_to(y, sizeof(T)))) return -10;
  Launch l;
  if (int st = make_launch(ctx, &l)) return st;
  if (n == 0) return B2_STATUS_OK;
  B2_DBG_RANGE(l, a, (size_t)((n - 1) * lda + n) * sizeof(T));
  B2_DBG_VEC(l, x, n, incx);
  B2_DBG_VEC(l, y, n, incy);
  B2_DBG_COMMIT(l);
  if (alpha == T(0)) return scale_y<T>(l, y, incy, n, beta);
  L2Args<T> args = {};
  args.a = a;
  args.lda = lda;
  args.rows = args.cols = n;
  args.xc = args.xr = vec_base(x, n, incx);
  args.incxc = args.incxr = incx;
  args.alpha = alpha;
  args.beta = beta;
  args.y = vec_base(y, n, incy);
  args.incy = incy;
  // the stored triangle as it sits in the row-major view of the buffer
  const bool upper = (order == B2_ROW_MAJOR) == (uplo == B2_UPPER);
  const L2Plan plan = plan_tri(args);
  if (knob(kKnobTriTile) == 1 || knob(kKnobGather) >= 2) {  // (a forced tile kernel stays forced)
    bool handled = false;
    const bool room = tri_room(l, args, plan, true);
    const int st = upper ? ga::run<T, Kind<true, true, TRI_UPPER, false, true>>(l, args, &handled, false, room)
                         : ga::run<T, Kind<true, true, TRI_LOWER, false, true>>(l, args, &handled, false, room);
    if (handled) return st;
  }
  // The tile kernel with the shared-memory ring (16-byte aligned matrices) is the faster one while the triangle is small:
  // its persistent blocks start at once, the general tile kernel streams faster.  Upper and lower triangle in turn,
  // general / ring, us for the pair: float n = 4096 25.0 / 23.5, 4608 (40 MiB) 26.9 / 27.1, 4800 (44) 27.4 / 31.1, 5792 33.8 / 39.4,
  // 8192 53.2 / 56.3; double n = 3008 24.8 / 24.6, 4096 (64) 33.1 / 35.5, 4352 (72) 36.0 / 39.2, 5008 44.9 / 49.1, 8192 99.3 /
  // 103.8.  (The line in double is from before tri_rows, when 4096 took 37.9 / 36.7.)
  // Knob value 2 forces the ring kernel at every size (tests).
  const bool small = (double)n * (double)n * sizeof(T) / 2 <= symv_ring_bytes(sizeof(T));
  if (knob(kKnobTriTile) == 2 || (knob(kKnobTriTile) == 1 && small)) {
    bool handled = false;
    const int st = upper ? tt::tri_tile_run<T, true, true, TRI_UPPER, false, true>(l, a, lda, n, args.xc, incx, alpha, beta,
                                                                                  args.y, incy, &handled)
                         : tt::tri_tile_run<T, true, true, TRI_LOWER, false, true>(l, a, lda, n, args.xc, incx, alpha, beta,
                                                                                  args.y, incy, &handled);
    if (handled) return st;
  }
  if (upper) return l2_dispatch<T, Kind<true, true, TRI_UPPER, false, true>, false>(l, args, plan, false);
  return l2_dispatch<T, Kind<true, true, TRI_LOWER, false, true>, false>(l, args, plan, false);
}

template <typename T, bool ROW, int TRI>
static int trmv_kind(const Launch& l, const L2Args<T>& args, bool unit) {
  // (column tiles of 128 elements, of 64 in double on aligned matrices: plan_colout)
  const bool narrow = sizeof(T) == 8 && aligned_to(args.a, 16) && args.lda % VecLen<T>::value == 0;
  const L2Plan plan = ROW ? plan_rowout(args, false, kShortRowsTrmv) : plan_colout(args, false, tri_rows(args, narrow ? 64 : 128));
  if constexpr (!ROW) {
    if (knob(kKnobTriTile) == 1 || knob(kKnobGather) >= 2) {
      bool handled = false;
      const bool room = tri_room(l, args, plan, false);
      const int st = unit ? ga::run<T, Kind<false, true, TRI, true, false>>(l, args, &handled, false, room)
                          : ga::run<T, Kind<false, true, TRI, false, false>>(l, args, &handled, false, room);
      if (handled) return st;
    }
  }
  if constexpr (ROW) {
    if ((knob(kKnobTriTile) == 1 && knob(kKnobGather) != 0) || knob(kKnobGather) >= 2) {  // (a forced tile kernel stays forced)
      bool handled = false;
      const int st = ts::run<T, TRI>(l, args, unit, &handled);
      if (handled) return st;
    }
  }
  // The tile kernel with the shared-memory ring serves trmv where it measured faster than the
  // general tile kernel: float row sums with a strided x (knob value 2: always, for the tests).
  const bool ring = knob(kKnobTriTile) == 2 || (knob(kKnobTriTile) == 1 && sizeof(T) == 4 && ROW && args.incxc != 1);
  if (ring) {
    bool handled = false;
    const int st =
        unit ? tt::tri_tile_run<T, ROW, !ROW, TRI, true, false>(l, args.a, args.lda, args.rows, args.xc, args.incxc, T(1), T(0),
                                                               args.y, args.incy, &handled)
             : tt::tri_tile_run<T, ROW, !ROW, TRI, false, false>(l, args.a, args.lda, args.rows, args.xc, args.incxc, T(1), T(0),
                                                                args.y, args.incy, &handled);
    if (handled) return st;
  }
  if (unit) return l2_dispatch<T, Kind<ROW, !ROW, TRI, true, false>, false>(l, args, plan, false);
  return l2_dispatch<T, Kind<ROW, !ROW, TRI, false, false>, false>(l, args, plan, false);
}

template <typename T>
static int trmv_impl(const b2_ctx* ctx, int order, int uplo, int trans, int diag, int64_t n, const T* a, int64_t lda,
                     T* x, int64_t incx) {
  if (int e = check_square(order, n, a, lda, 1, 5, 6, 7)) return e;
  if (uplo != B2_UPPER && uplo != B2_LOWER) return -2;
  if (trans != B2_NO_TRANS && trans != B2_TRANS) return -3;
  if (diag != B2_NON_UNIT && diag != B2_UNIT) return -4;
  if (incx == 0) return -9;
  if (n > 0 && (x == nullptr || !aligned_to(x, sizeof(T)))) return -8;
  Launch l;
  if (int st = make_launch(ctx, &l)) return st;
  if (n == 0) return B2_STATUS_OK;
  B2_DBG_RANGE(l, a, (size_t)((n - 1) * lda + n) * sizeof(T));
  B2_DBG_VEC(l, x, n, incx);
  B2_DBG_COMMIT(l);
  L2Args<T> args = {};
  args.a = a;
  args.lda = lda;
  args.rows = args.cols = n;
  args.xc = args.xr = vec_base(x, n, incx);
  args.incxc = args.incxr = incx;
  args.alpha = T(1);
  args.beta = T(0);
  args.y = vec_base(x, n, incx);
  args.incy = incx;
  const bool upper = (order == B2_ROW_MAJOR) == (uplo == B2_UPPER);
  const bool row = (order == B2_ROW_MAJOR) == (trans == B2_NO_TRANS);
  const bool unit = diag == B2_UNIT;
  if (row) return upper ? trmv_kind<T, true, TRI_UPPER>(l, args, unit) : trmv_kind<T, true, TRI_LOWER>(l, args, unit);
  return upper ? trmv_kind<T, false, TRI_UPPER>(l, args, unit) : trmv_kind<T, false, TRI_LOWER>(l, args, unit);
}

}  // namespace b2
