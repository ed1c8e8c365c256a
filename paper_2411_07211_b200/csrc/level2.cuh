// Level-2 matrix-vector template layer (Section 6.2.2 of the paper).
//
// One tile kernel serves gemv (N and T), symv and trmv in every option combination.  The
// matrix is always seen in its canonical row-major view (rows x cols, row stride lda; a
// column-major call is the transposed row-major problem).  A thread block owns a band of
// rows and a range of column tiles and may produce
//   ROWOUT: rowacc_i = sum_j A_ij * xc_j   (each row is a contiguous dot product), and/or
//   COLOUT: colacc_j = sum_i A_ij * xr_i   (column sums accumulated in registers),
// restricted to the upper / lower triangle for the triangular kinds.  This is the paper's
// level-2 recipe restated for a GPU: several rows are processed at once so the x values sit in
// registers and are reused (unroll-and-jam), triangular bounds are rounded to tile
// boundaries so full tiles run unmasked and only diagonal tiles are predicated, and narrow
// matrices get shapes whose whole row fits the lanes of a warp (the "skinny" case).
//
// Blocks write either the final result (when no other block contributes to the same
// output) or a partial into the workspace; l2_finalize then adds the partials in a fixed
// order and applies alpha / beta.  No atomics: results are bit-reproducible.
#pragma once

#include <algorithm>

#include <type_traits>

#include "common.cuh"

namespace b2 {

enum { TRI_FULL = 0, TRI_UPPER = 1, TRI_LOWER = 2 };

template <bool ROWOUT_, bool COLOUT_, int TRI_, bool UNIT_, bool SYM_>
struct Kind {
  static constexpr bool ROWOUT = ROWOUT_, COLOUT = COLOUT_, UNIT = UNIT_, SYM = SYM_;
  static constexpr int TRI = TRI_;
};

// LPR lanes cover one row segment, so a warp covers G = 32/LPR rows per step; each lane owns
// CU packs of V columns; RU row steps are in flight per warp.
// NCT: column tiles a block of a COLOUT kind walks per row step (their column sums stay in
// registers side by side, the row sums run across all of them).
template <int LPR_, int CU_, int RU_, int NCT_ = 1>
struct Shape {
  static constexpr int LPR = LPR_, CU = CU_, RU = RU_, G = 32 / LPR_, NCT = NCT_;
  static constexpr int MINB = NCT_ == 1 ? 4 : 3;  // resident blocks per SM the register budget aims at
  static constexpr int RB = kWarps * G * RU_;  // rows per block step
  template <int V>
  static constexpr int tc() {
    return LPR_ * V * CU_;
  }
};

template <typename T>
struct L2Args {
  const T* a;
  int64_t lda, rows, cols;
  const T* xc;  // vector indexed by column (ROWOUT), base per vec_base()
  int64_t incxc;
  const T* xr;  // vector indexed by row (COLOUT)
  int64_t incxr;
  T* rowpart;  // [ncs][rows]
  T* colpart;  // [nrs][cols]
  T* colspill; // [nrs][nct][V - 1]: column sums left of a block's own columns (SHIFT)
  int64_t rows_per_cta;
  int ctiles_per_cta, nct, nrs, ncs;
  int direct;  // 1: blocks write alpha*acc + beta*y straight to y
  int xc_vec;  // xc is 16-byte aligned with increment 1 (value 1) or 2 (value 2): read it in packs
  T alpha, beta;
  T* y;
  int64_t incy;
};

// Which parts of the tile grid hold any element of the triangle.  Used identically by the
// tile kernel (to skip work) and by the finalize kernel (to know which partials exist).
template <int TRI>
__host__ __device__ __forceinline__ bool region_active(int64_t r0, int64_t r1, int64_t c0, int64_t c1) {
  if (TRI == TRI_UPPER) return c1 - 1 >= r0;  // some (i, j) with j >= i
  if (TRI == TRI_LOWER) return c0 <= r1 - 1;  // some (i, j) with j <= i
  return true;
}
// Tile lies strictly inside the triangle (no diagonal element, no masking needed).
template <int TRI>
__device__ __forceinline__ bool region_strictly_inside(int64_t r0, int64_t r1, int64_t c0, int64_t c1) {
  if (TRI == TRI_UPPER) return c0 >= r1;
  if (TRI == TRI_LOWER) return c1 <= r0;
  return true;
}

// SHIFT: rows that start off 16-byte boundaries, read in aligned packs all the same.  A warp's rows are congruent
// modulo 8 and 8 * lda is a multiple of V, so they all start the same number s of elements past a boundary; the warp
// takes its packs from s elements before the row on, and its column q of a tile is column q - s of the matrix.  Row
// sums do not mind; column sums of a tile cover its TC columns and the V - 1 before them, which go to colspill.  Only
// packs that the matrix edge cuts are read element by element.  (Element loads everywhere, four times the load
// instructions: float n = 8191 symv 60 us, trmv 34, gemv 54; aligned 28, 24, 43.)
template <typename T, int V, class K, class S, bool SHIFT>
__global__ void __launch_bounds__(kThreads, S::MINB) l2_tile_kernel(const L2Args<T> p) {
  constexpr int LPR = S::LPR, CU = S::CU, RU = S::RU, G = S::G, RB = S::RB;
  constexpr int TC = LPR * V * CU, SH = SHIFT ? V - 1 : 0;
  static_assert(!SHIFT || (G == 1 && S::NCT == 1), "a warp's rows are congruent modulo kWarps");
  constexpr int NCT = K::COLOUT ? S::NCT : 1;
  using P = Pack<T, V>;
  grid_dep_wait();
  grid_dep_launch();  // the next kernel of the stream (often this call's finalize pass) may be scheduled early

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane / LPR, q = lane % LPR;
  // Blocks start in index order.  In an upper triangle the bottom-right blocks are the ones that the
  // matrix edge cuts (the last column tile, ragged when n is not a multiple of the tile, is there the
  // LONGEST column); started last and running alone they would be the tail (measured in double at
  // n = 8190, column sums: 74 us against 48), so the order is reversed and the last block to start
  // is the small one in the top-left corner.
  const unsigned bidx = K::TRI == TRI_UPPER ? gridDim.x - 1u - blockIdx.x : blockIdx.x;
  const int cs = (int)(bidx % (unsigned)p.ncs);
  const int64_t rs = bidx / (unsigned)p.ncs;
  const int64_t r_begin = rs * p.rows_per_cta;
  const int64_t r_end = min(p.rows, r_begin + p.rows_per_cta);
  const int ct_begin = cs * p.ctiles_per_cta;
  const int ct_end = min(p.nct, ct_begin + p.ctiles_per_cta);
  const int64_t c_lo = (int64_t)ct_begin * TC, c_hi = min(p.cols, (int64_t)ct_end * TC);
  if (!region_active<K::TRI>(r_begin, r_end, c_lo - SH, c_hi)) return;

  T colacc[NCT][CU][V];
  T xcv[NCT][CU][V];
  int xcv_ct[NCT];  // column tile whose x values are in xcv[c]
#pragma unroll
  for (int c = 0; c < NCT; ++c) {
    xcv_ct[c] = -1;
#pragma unroll
    for (int u = 0; u < CU; ++u)
#pragma unroll
      for (int e = 0; e < V; ++e) colacc[c][u][e] = T(0), xcv[c][u][e] = T(0);
  }

  // Address arithmetic is hoisted: inside a tile everything is a 32-bit local index or a
  // pointer bumped by a precomputed stride.
  const int lrow0 = warp * G + g;                            // first local row of this thread
  const int64_t rstride = (int64_t)kWarps * G * p.lda;       // elements between a thread's rows
  const int64_t xstride = (int64_t)kWarps * G * p.incxr;
  const int s = SHIFT ? (int)(((unsigned long long)p.a / sizeof(T) + (unsigned long long)lrow0 * (unsigned long long)p.lda) % V) : 0;
  const T* a_cta = p.a + (r_begin + lrow0) * p.lda + (q * V - s);  // row r_begin + lrow0, column q*V (- s)

  auto load_xc = [&](T (&xv_)[CU][V], int64_t c0) {  // x values of the column tile at c0
    if (SHIFT && c0 > 0 && c0 + TC <= p.cols) {
      const T* xp = p.xc + (c0 + q * V - s) * p.incxc;
#pragma unroll
      for (int u = 0; u < CU; ++u)
#pragma unroll
        for (int e = 0; e < V; ++e) xv_[u][e] = __ldg(xp + (u * LPR * V + e) * p.incxc);
    } else if (SHIFT) {
#pragma unroll
      for (int u = 0; u < CU; ++u)
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const int64_t j = c0 + (u * LPR + q) * V + e - s;
          xv_[u][e] = j >= 0 && j < p.cols ? __ldg(p.xc + j * p.incxc) : T(0);
        }
    } else if (V > 1 && p.xc_vec == 1 && c0 + TC <= p.cols) {
#pragma unroll
      for (int u = 0; u < CU; ++u) {
        const P xv = ld_ro<T, V>(p.xc + c0 + (u * LPR + q) * V);
#pragma unroll
        for (int e = 0; e < V; ++e) xv_[u][e] = xv.v[e];
      }
    } else if (V > 1 && p.xc_vec == 2 && c0 + TC < p.cols) {
      // increment 2: the V values sit in two consecutive packs (even positions); the odd
      // position after the last value exists because the tile is not the vector's last
#pragma unroll
      for (int u = 0; u < CU; ++u) {
        const T* xp = p.xc + 2 * (c0 + (u * LPR + q) * V);
        const P x0 = ld_ro<T, V>(xp), x1 = ld_ro<T, V>(xp + V);
#pragma unroll
        for (int e = 0; e < V; ++e) xv_[u][e] = (2 * e < V) ? x0.v[(2 * e) % V] : x1.v[(2 * e) % V];
      }
    } else {
#pragma unroll
      for (int u = 0; u < CU; ++u)
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const int64_t j = c0 + (u * LPR + q) * V + e;
          xv_[u][e] = j < p.cols ? __ldg(p.xc + j * p.incxc) : T(0);
        }
    }
  };

  // Column-sum kinds: the row steps that lie whole inside the matrix and the triangle run in a loop of their own,
  // with pointers that advance and no tests: 64-bit bounds and addresses per step were 2/3 of the instructions.
  // (gemv, both products of a 16384 matrix, 328 -> 308 us in float, 670 -> 606 in double; symv n = 16384 190 -> 181,
  // trmv n = 4096 in double 34 -> 31.  Not for shifted float rows, which spill here: symv n = 8191 72 -> 77 us.)
  constexpr bool STEADY = K::COLOUT && NCT == 1 && !(SHIFT && sizeof(T) == 4);
  // CUT: the last column tile of an upper triangle, which is its longest column, takes part when the matrix edge cuts it,
  // its loads under predicates that do not change along the way.  A step in the general form below lasts half a
  // microsecond longer here than it does in a kernel without this loop, and with every step of that column in it these
  // blocks were the tail of the launch: trmv in double, n = 5360, 26.2 us without any such loop, 30.0 with the loop
  // for whole tiles only, 25.4 so; n = 3008 in float 14.9 -> 9.6; symv in float, n = 7400, 28.4, 30.9, 24.4.
  // With shifted packs the first tile of a lower triangle, its longest column, is cut as well, by the beginning of the
  // rows: symv in double, n = 4001, upper / lower, by elements 26.3 / 25.5, in shifted packs 26.6 / 28.4, 21.5 / 23.0 so.
  constexpr bool CUT = STEADY && (K::TRI == TRI_UPPER || (SHIFT && K::TRI == TRI_LOWER));
  constexpr bool CUT_FIRST = CUT && K::TRI == TRI_LOWER;
  int64_t fast_lo = 0, fast_hi = 0;  // first row of the first such step, end of the last
  if constexpr (STEADY) {
    if (CUT || (c_lo + TC <= p.cols && (!SHIFT || c_lo > 0))) {
      fast_lo = r_begin, fast_hi = r_end;
      if (K::TRI == TRI_LOWER) fast_lo = max(r_begin, (c_lo + TC - 1) / RB * RB + RB);  // (rows past the last column)
      if (K::TRI == TRI_UPPER) fast_hi = min(r_end, c_lo - SH);
      fast_hi = fast_hi > fast_lo ? fast_lo + (fast_hi - fast_lo) / RB * RB : fast_lo;
    }
  }
  for (int64_t rb = r_begin; rb < r_end; rb += RB) {
    if constexpr (STEADY) {
      if (rb == fast_lo && fast_hi > fast_lo) {
        const int nst = (int)((fast_hi - fast_lo) / RB);
        const T* at = a_cta + (fast_lo - r_begin) * p.lda + c_lo;
        const T* xp = p.xr + (fast_lo + lrow0) * p.incxr;
        const int64_t astep = (int64_t)RB * p.lda, xstep = (int64_t)RB * p.incxr;
        constexpr int LPV = LPR / RU;
        T* rp = p.rowpart + (int64_t)cs * p.rows + fast_lo + ((q / LPV) * kWarps + warp) * G + g;
        if (K::ROWOUT && xcv_ct[0] != ct_begin) {
          xcv_ct[0] = ct_begin;
          load_xc(xcv[0], c_lo);
        }
        if constexpr (CUT) {
          if (CUT_FIRST ? c_lo == 0 : c_lo + TC > p.cols) {
            const int nc = (int)min((int64_t)(TC + SH), p.cols - c_lo);  // columns that exist (CUT_FIRST: from 0 on)
            auto cut_steps = [&](auto packs) {    // in whole packs, or by elements
#pragma unroll 1
              for (int st = 0; st < nst; ++st) {
                P av[RU][CU];
                T xv[RU];
#pragma unroll
                for (int ru = 0; ru < RU; ++ru)
#pragma unroll
                  for (int u = 0; u < CU; ++u) {
                    const T* ap = at + ru * rstride + u * (LPR * V);
                    const int lc = (u * LPR + q) * V - s;
                    if constexpr (decltype(packs)::value) av[ru][u] = ld_nc_if<T, V>(ap, lc < nc);
                    else {
#pragma unroll
                      for (int e = 0; e < V; ++e) av[ru][u].v[e] = ld_el_if<T>(ap + e, CUT_FIRST ? lc + e >= 0 : lc + e < nc);
                    }
                  }
#pragma unroll
                for (int ru = 0; ru < RU; ++ru) xv[ru] = __ldg(xp + ru * xstride);
                at += astep;
                xp += xstep;
                T racc[RU];
#pragma unroll
                for (int ru = 0; ru < RU; ++ru) {
                  racc[ru] = T(0);
#pragma unroll
                  for (int u = 0; u < CU; ++u)
#pragma unroll
                    for (int e = 0; e < V; ++e) {
                      if (K::ROWOUT) racc[ru] = av[ru][u].v[e] * xcv[0][u][e] + racc[ru];
                      colacc[0][u][e] = av[ru][u].v[e] * xv[ru] + colacc[0][u][e];
                    }
                }
                if (K::ROWOUT) {
                  const T sum = multi_group_sum<LPR, RU>(racc, lane);
                  if (q % LPV == 0) *rp = sum;
                  rp += RB;
                }
              }
            };
            if (!SHIFT && nc % V == 0) cut_steps(std::bool_constant<!SHIFT>());
            else cut_steps(std::false_type());
            rb = fast_hi - RB;
            continue;
          }
        }
#pragma unroll 1
        for (int st = 0; st < nst; ++st) {
          P av[RU][CU];
          T xv[RU];
#pragma unroll
          for (int ru = 0; ru < RU; ++ru)
#pragma unroll
            for (int u = 0; u < CU; ++u) av[ru][u] = ld_nc<T, V>(at + ru * rstride + u * (LPR * V));
#pragma unroll
          for (int ru = 0; ru < RU; ++ru) xv[ru] = __ldg(xp + ru * xstride);
          at += astep;
          xp += xstep;
          T racc[RU];
#pragma unroll
          for (int ru = 0; ru < RU; ++ru) {
            racc[ru] = T(0);
#pragma unroll
            for (int u = 0; u < CU; ++u)
#pragma unroll
              for (int e = 0; e < V; ++e) {
                if (K::ROWOUT) racc[ru] = av[ru][u].v[e] * xcv[0][u][e] + racc[ru];
                colacc[0][u][e] = av[ru][u].v[e] * xv[ru] + colacc[0][u][e];
              }
          }
          if (K::ROWOUT) {
            const T sum = multi_group_sum<LPR, RU>(racc, lane);
            if (q % LPV == 0) *rp = sum;
            rp += RB;
          }
        }
        rb = fast_hi - RB;
        continue;
      }
    }
    const int64_t rb_end = min(rb + RB, r_end);
    if (!region_active<K::TRI>(rb, rb_end, c_lo - SH, c_hi)) continue;
    const int nr = (int)(rb_end - rb);  // rows of this batch
    const T* a_rb = a_cta + (rb - r_begin) * p.lda;
    T rowacc[RU], xrv[RU];
#pragma unroll
    for (int ru = 0; ru < RU; ++ru) {
      rowacc[ru] = T(0);
      xrv[ru] = T(0);
    }
    if (K::COLOUT) {
      const T* xp = p.xr + (rb + lrow0) * p.incxr;
#pragma unroll
      for (int ru = 0; ru < RU; ++ru)
        if (lrow0 + ru * kWarps * G < nr) xrv[ru] = __ldg(xp + ru * xstride);
    }
    // COLOUT kinds: slot c holds column tile ct_begin + c; ROWOUT-only kinds: one slot, any
    // number of column tiles.
#pragma unroll
    for (int c = 0; c < NCT; ++c) {
    const int ct_lo = K::COLOUT ? ct_begin + c : ct_begin;
    const int ct_hi = K::COLOUT ? min(ct_lo + 1, ct_end) : ct_end;
    for (int ct = ct_lo; ct < ct_hi; ++ct) {
      const int64_t c0 = (int64_t)ct * TC, c1 = min(p.cols, c0 + TC);
      if (!region_active<K::TRI>(rb, rb_end, c0 - SH, c1)) continue;
      if (K::ROWOUT && xcv_ct[c] != ct) {
        xcv_ct[c] = ct;
        load_xc(xcv[c], c0);
      }
      const bool fast = !STEADY && (rb + RB <= r_end) && (c0 + TC <= p.cols) && (!SHIFT || c0 > 0) &&
                        region_strictly_inside<K::TRI>(rb, rb + RB, c0 - SH, c0 + TC);
      if (fast) {
        P av[RU][CU];
        const T* at = a_rb + c0;
#pragma unroll
        for (int ru = 0; ru < RU; ++ru)
#pragma unroll
          for (int u = 0; u < CU; ++u) av[ru][u] = ld_nc<T, V>(at + ru * rstride + u * (LPR * V));
#pragma unroll
        for (int ru = 0; ru < RU; ++ru)
#pragma unroll
          for (int u = 0; u < CU; ++u)
#pragma unroll
            for (int e = 0; e < V; ++e) {
              if (K::ROWOUT) rowacc[ru] = av[ru][u].v[e] * xcv[c][u][e] + rowacc[ru];
              if (K::COLOUT) colacc[c][u][e] = av[ru][u].v[e] * xrv[ru] + colacc[c][u][e];
            }
      } else if (!SHIFT && K::TRI == TRI_FULL && (V == 1 || (c1 - c0) % V == 0)) {
        // gemv: a tile that the matrix edge cuts (fewer rows than RB, or a row that ends on a
        // pack boundary before the tile does): the loads still go out together, each under its
        // own row / pack predicate.  Narrow matrices (fewer columns than one tile) and short
        // ones (fewer rows than one step) live entirely here.  A masked pack is zero and meets
        // a zero x value, so it adds nothing.
        const int npk = (int)(c1 - c0) / V;  // packs of this tile that exist
        P av[RU][CU];
        const T* at = a_rb + c0;
#pragma unroll
        for (int ru = 0; ru < RU; ++ru) {
          const bool rok = lrow0 + ru * kWarps * G < nr;
#pragma unroll
          for (int u = 0; u < CU; ++u) {
#pragma unroll
            for (int e = 0; e < V; ++e) av[ru][u].v[e] = T(0);
            if (rok && u * LPR + q < npk) av[ru][u] = ld_nc<T, V>(at + ru * rstride + u * (LPR * V));
          }
        }
#pragma unroll
        for (int ru = 0; ru < RU; ++ru)
#pragma unroll
          for (int u = 0; u < CU; ++u)
#pragma unroll
            for (int e = 0; e < V; ++e) {
              if (K::ROWOUT) rowacc[ru] = av[ru][u].v[e] * xcv[c][u][e] + rowacc[ru];
              if (K::COLOUT) colacc[c][u][e] = av[ru][u].v[e] * xrv[ru] + colacc[c][u][e];
            }
      } else {
        // Diagonal tiles and column edges inside a pack: local 32-bit indices; d = (first column)
        // - (first row), so element (li, lj) lies on the diagonal when d + lj == li.  All loads
        // of the tile go out together, each under its own predicate (a pack wholly outside the
        // triangle or the matrix is not read), and only then are the elements masked: loads
        // issued one by one between the branches made such a tile last several memory latencies.
        const int64_t d64 = c0 - rb;
        const int d = (int)(d64 > (1 << 24) ? (1 << 24) : d64 < -(1 << 24) ? -(1 << 24) : d64);
        const int nc = (int)(p.cols - c0 < TC + SH ? p.cols - c0 : TC + SH);  // local columns that exist (of those before the tile: SHIFT)
        const int lo = SHIFT && c0 == 0 ? 0 : -SH;                            // first local column that exists
        const T* at = a_rb + c0;
        P av[RU][CU];
#pragma unroll
        for (int ru = 0; ru < RU; ++ru) {
          const int li = lrow0 + ru * kWarps * G;
#pragma unroll
          for (int u = 0; u < CU; ++u) {
            const int lc = (u * LPR + q) * V - s;
            bool use = li < nr && lc < nc;
            if (K::TRI == TRI_UPPER) use = use && d + lc + V - 1 >= li;
            if (K::TRI == TRI_LOWER) use = use && d + lc <= li;
            av[ru][u] = ld_nc_if<T, V>(at + ru * rstride + u * (LPR * V), use && (V == 1 || (lc + V <= nc && (!SHIFT || lc >= lo))));
          }
        }
        if (V > 1 && (SHIFT || nc % V != 0)) {  // the rows start or end inside a pack: that pack element by element
#pragma unroll
          for (int u = 0; u < CU; ++u) {
            const int lc = (u * LPR + q) * V - s;
            if (lc < nc && (lc + V > nc || (SHIFT && lc < lo))) {  // (one branch; the loads below are predicated, not branched)
#pragma unroll
              for (int ru = 0; ru < RU; ++ru) {
                const int li = lrow0 + ru * kWarps * G;
                bool use = li < nr;
                if (K::TRI == TRI_UPPER) use = use && d + lc + V - 1 >= li;
                if (K::TRI == TRI_LOWER) use = use && d + lc <= li;
                const T* ap = at + ru * rstride + u * (LPR * V);
#pragma unroll
                for (int e = 0; e < V; ++e) av[ru][u].v[e] = ld_el_if<T>(ap + e, use && lc + e < nc && (!SHIFT || lc + e >= lo));
              }
            }
          }
        }
#pragma unroll
        for (int ru = 0; ru < RU; ++ru) {
          const int li = lrow0 + ru * kWarps * G;
#pragma unroll
          for (int u = 0; u < CU; ++u) {
            const int lc = (u * LPR + q) * V - s;
#pragma unroll
            for (int e = 0; e < V; ++e) {
              const int lj = lc + e;
              bool in = li < nr && lj < nc && (!SHIFT || lj >= lo);
              if (K::TRI == TRI_UPPER) in = in && d + lj >= li;
              if (K::TRI == TRI_LOWER) in = in && d + lj <= li;
              const bool dg = (K::TRI != TRI_FULL) && (d + lj == li);
              const T v = (K::UNIT && dg) ? T(1) : av[ru][u].v[e];
              // (a select, not a product with zero: x may hold infinities where the triangle ends)
              if (K::ROWOUT) rowacc[ru] = in ? v * xcv[c][u][e] + rowacc[ru] : rowacc[ru];
              if (K::COLOUT && !(K::SYM && dg)) colacc[c][u][e] = in ? v * xrv[ru] + colacc[c][u][e] : colacc[c][u][e];
            }
          }
        }
      }
    }
    }  // slot c
    if (K::ROWOUT) {  // all RU row sums in one transposing butterfly
      constexpr int LPV = LPR / RU;  // lanes left per row after the reduction
      const T sum = multi_group_sum<LPR, RU>(rowacc, lane);
      const int64_t i = rb + ((q / LPV) * kWarps + warp) * G + g;
      if (q % LPV == 0 && i < r_end) {
        if (p.direct) {
          T* yp = p.y + i * p.incy;
          B2_STORE(yp, p.beta != T(0) ? p.alpha * sum + p.beta * *yp : p.alpha * sum);
        } else {
          p.rowpart[(int64_t)cs * p.rows + i] = sum;
        }
      }
    }
  }

  if constexpr (K::COLOUT) {  // NCT column tiles per block for these kinds
    __shared__ T sm[kWarps][NCT * TC + SH];  // SHIFT: entry t is column c_lo - SH + t
    if (SHIFT && lane < SH) sm[warp][lane < SH - s ? lane : TC + lane] = T(0);
#pragma unroll
    for (int c = 0; c < NCT; ++c)
#pragma unroll
      for (int u = 0; u < CU; ++u)
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const T sum = cross_group_sum<LPR>(colacc[c][u][e]);
          if (g == 0) sm[warp][c * TC + (u * LPR + q) * V + e + SH - s] = sum;
        }
    __syncthreads();
    for (int t = threadIdx.x; t < NCT * TC + SH; t += kThreads) {
      const int64_t j = c_lo - SH + t;
      if (j >= p.cols) break;
      T s = sm[0][t];
#pragma unroll
      for (int w = 1; w < kWarps; ++w) s += sm[w][t];
      if (SHIFT && t < SH) {
        p.colspill[(rs * p.nct + cs) * SH + t] = s;
      } else if (p.direct) {
        T* yp = p.y + j * p.incy;
        B2_STORE(yp, p.beta != T(0) ? p.alpha * s + p.beta * *yp : p.alpha * s);
      } else {
        p.colpart[rs * p.cols + j] = s;
      }
    }
  }
}

// Adds the partials of each output in a fixed order and writes y = alpha*sum + beta*y.
// A block handles 256/SLICES consecutive outputs; SLICES threads share one output and split
// its list of partials (slice k takes partials k, k+SLICES, ...), then combine through shared
// memory in slice order.  Launched as a programmatic dependent of the tile kernel.
// SH: columns before its own that a tile of the first pass covers (SHIFT: V - 1, else 0).
template <typename T, class K, int SLICES>
__global__ void __launch_bounds__(kThreads) l2_finalize(const L2Args<T> p, int RB, int TC, int SH) {
  constexpr int OUTB = kThreads / SLICES;
  __shared__ T sm[SLICES][OUTB];
  grid_dep_wait();
  grid_dep_launch();
  const int o = threadIdx.x % OUTB, slice = threadIdx.x / OUTB;
  const int64_t nout = K::ROWOUT ? p.rows : p.cols;
  const int64_t i = (int64_t)blockIdx.x * OUTB + o;
  T s = T(0);
  // This slice's share of the partials [lo, hi) of a list with the given stride: four loads in flight, added in order.
  // (Which partials of a triangle exist is a few 32-bit divisions per output; tested one by one, in 64-bit arithmetic,
  // it was half of the kernel's instructions: symv of n = 8192 in double 113.3 us, so 110.)
  using I = typename std::conditional<K::TRI == TRI_FULL, int64_t, unsigned>::type;
  auto add_partials = [&](T sum, const T* list, int64_t stride, int lo, int hi) -> T {
    int k = lo + slice;
    const T* ptr = list + (int64_t)k * stride;
    const int64_t step = stride * SLICES;
    for (; k + 3 * SLICES < hi; k += 4 * SLICES, ptr += 4 * step) {
      const T v0 = __ldcg(ptr), v1 = __ldcg(ptr + step), v2 = __ldcg(ptr + 2 * step), v3 = __ldcg(ptr + 3 * step);
      sum += v0, sum += v1, sum += v2, sum += v3;
    }
    for (; k < hi; k += SLICES, ptr += step) sum += __ldcg(ptr);
    return sum;
  };
  if (i < nout) {
    if (K::ROWOUT) {
      const I span = (I)TC * p.ctiles_per_cta;
      const I rb = (I)i - (I)i % (I)RB, rb_end = min((I)p.rows, rb + (I)RB);  // (rows_per_cta is a multiple of RB)
      const int lo = K::TRI == TRI_UPPER ? (int)(rb / span) : 0;
      const int hi = K::TRI == TRI_LOWER ? min(p.ncs, (int)((rb_end - 1 + SH) / span) + 1) : p.ncs;
      s = add_partials(s, p.rowpart + i, p.rows, lo, hi);
    }
    if (K::COLOUT) {
      const I span = (I)TC * p.ctiles_per_cta, rpc = (I)p.rows_per_cta;  // columns and rows of one block
      const I ct = (I)i / span, c_lo = ct * span;
      auto first = [&](I c) { return K::TRI == TRI_LOWER && c > (I)SH ? (int)((c - SH) / rpc) : 0; };
      auto last = [&](I c) { return K::TRI == TRI_UPPER ? min((int)p.nrs, (int)((min((I)p.cols, c) - 1) / rpc) + 1) : (int)p.nrs; };
      s = add_partials(s, p.colpart + i, p.cols, first(c_lo), last(c_lo + span));
      if (SH > 0 && (I)i - c_lo >= span - SH && (int64_t)ct + 1 < p.nct)  // the next tile's share of the last columns
        s = add_partials(s, p.colspill + ((int64_t)ct + 1) * SH + ((I)i - c_lo - (span - SH)), (int64_t)p.nct * SH,
                         first(c_lo + span), last(c_lo + 2 * span));
    }
  }
  if (SLICES > 1) {
    sm[slice][o] = s;
    __syncthreads();
    if (slice != 0) return;
#pragma unroll
    for (int k = 1; k < SLICES; ++k) s += sm[k][o];
  }
  if (i < nout) {
    T* yp = p.y + i * p.incy;
    B2_STORE(yp, p.beta != T(0) ? p.alpha * s + p.beta * *yp : p.alpha * s);
  }
}

// y <- beta*y (alpha == 0 shortcut); beta == 0 writes zeros without reading.
template <typename T>
__global__ void __launch_bounds__(kThreads) l2_scale_y(T* y, int64_t incy, int64_t n, T beta) {
  grid_dep_wait();
  grid_dep_launch();
  const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  if (i < n) y[i * incy] = beta == T(0) ? T(0) : beta * y[i * incy];
}

// ------------------------------------------------------------------------------- host side
struct L2Plan {
  int shape;             // index into the shape table
  int tile_cols;         // columns of a column tile
  int64_t rows_per_cta;  // multiple of the shape's RB
  int ctiles_per_cta;
};

template <typename T, class K, int SLICES>
static void launch_finalize(const Launch& l, const L2Args<T>& args, int RB, int TC, int64_t nout, int SH = 0) {
  constexpr int OUTB = kThreads / SLICES;
  launch_chained(l2_finalize<T, K, SLICES>, dim3((unsigned)((nout + OUTB - 1) / OUTB)), dim3(kThreads), 0, l.stream, args, RB, TC, SH);
}

// Launches the tile kernel (+ finalize when partials are needed) for one shape.
template <typename T, int V, class K, class S, bool SHIFT = false>
static int l2_launch_shape(const Launch& l, L2Args<T> args, int64_t rows_per_cta, int ctiles_per_cta,
                           bool allow_direct) {
  constexpr int TC = S::template tc<V>();
  constexpr int RB = S::RB, SH = SHIFT ? V - 1 : 0;
  args.nct = (int)((args.cols + SH + TC - 1) / TC);
  args.xc_vec = (!SHIFT && K::ROWOUT && V > 1 && aligned_to(args.xc, 16)) ? (args.incxc == 1 ? 1 : args.incxc == 2 ? 2 : 0) : 0;
  if (K::COLOUT) ctiles_per_cta = S::NCT;
  if (ctiles_per_cta < 1) ctiles_per_cta = 1;
  if (ctiles_per_cta > args.nct) ctiles_per_cta = args.nct;
  rows_per_cta = ((rows_per_cta + RB - 1) / RB) * RB;
  if (rows_per_cta < RB) rows_per_cta = RB;
  for (;;) {  // shrink the number of partials until they fit the workspace
    args.rows_per_cta = rows_per_cta;
    args.ctiles_per_cta = ctiles_per_cta;
    args.nrs = (int)((args.rows + rows_per_cta - 1) / rows_per_cta);
    args.ncs = (args.nct + ctiles_per_cta - 1) / ctiles_per_cta;
    const bool single = (!K::ROWOUT || args.ncs == 1) && (!K::COLOUT || (args.nrs == 1 && !SHIFT)) && !(K::ROWOUT && K::COLOUT);
    args.direct = allow_direct && single;
    if (args.direct) break;
    size_t need = 0;
    if (K::ROWOUT) need += (size_t)args.ncs * args.rows * sizeof(T);
    const size_t row_bytes = (need + 255) / 256 * 256;
    const size_t col_bytes = ((K::COLOUT ? (size_t)args.nrs * args.cols * sizeof(T) : 0) + 255) / 256 * 256;
    if (K::COLOUT) need = row_bytes + (SHIFT ? col_bytes + (size_t)args.nrs * args.nct * SH * sizeof(T) : (size_t)args.nrs * args.cols * sizeof(T));
    if (need <= l.scratch_bytes) {
      args.rowpart = reinterpret_cast<T*>(l.scratch);
      args.colpart = reinterpret_cast<T*>(l.scratch + row_bytes);
      args.colspill = reinterpret_cast<T*>(l.scratch + row_bytes + col_bytes);
      break;
    }
    // (a block of a column-sum kind walks exactly S::NCT column tiles -- their sums sit in its
    // registers -- so only its row band can grow; a row-dot kind merges column splits)
    bool changed = false;
    if (K::ROWOUT && !K::COLOUT && ctiles_per_cta < args.nct) ctiles_per_cta *= 2, changed = true;
    if (ctiles_per_cta > args.nct) ctiles_per_cta = args.nct;
    if (K::COLOUT && rows_per_cta < args.rows) rows_per_cta *= 2, changed = true;
    if (!changed) return B2_STATUS_WORKSPACE_TOO_SMALL;
  }
  const int64_t nblocks = (int64_t)args.nrs * args.ncs;
  if (nblocks > 0x7fffffff) return B2_STATUS_NOT_IMPLEMENTED;
  launch_chained(l2_tile_kernel<T, V, K, S, SHIFT>, dim3((unsigned)nblocks), dim3(kThreads), 0, l.stream, args);
  if (int st = check_launch()) return st;
  if (!args.direct) {
    const int64_t nout = K::ROWOUT ? args.rows : args.cols;
    const int nparts = (K::ROWOUT ? args.ncs : 0) + (K::COLOUT ? args.nrs : 0);
    if (nparts >= 512) launch_finalize<T, K, 32>(l, args, RB, TC, nout, SH);
    else if (nparts >= 12) launch_finalize<T, K, 8>(l, args, RB, TC, nout, SH);
    else launch_finalize<T, K, 1>(l, args, RB, TC, nout, SH);
    if (int st = check_launch()) return st;
  }
  return B2_STATUS_OK;
}

// Shape table shared by all kinds.
using ShapeWide = Shape<32, 4, 2>;    // 2 KiB row segments, 16 rows per step
using ShapeWide4 = Shape<32, 4, 4>;   // the same, 32 rows per step
using ShapeMid = Shape<32, 1, 8>;     // 512 B row segments, 64 rows per step
using ShapeHalf = Shape<16, 1, 8>;    // 256 B row segments, 128 rows per step
using ShapeQuarter = Shape<8, 1, 8>;  // 128 B row segments, 256 rows per step
enum { SHAPE_WIDE = 0, SHAPE_MID = 1, SHAPE_HALF = 2, SHAPE_QUARTER = 3, SHAPE_WIDE4 = 4 };

inline int shape_rb(int shape) {
  switch (shape) {
    case SHAPE_WIDE: return ShapeWide::RB;
    case SHAPE_WIDE4: return ShapeWide4::RB;
    case SHAPE_MID: return ShapeMid::RB;
    case SHAPE_HALF: return ShapeHalf::RB;
    default: return ShapeQuarter::RB;
  }
}
inline int shape_packs_per_row(int shape) {  // packs of one row segment
  switch (shape) {
    case SHAPE_WIDE:
    case SHAPE_WIDE4: return 128;
    case SHAPE_MID: return 32;
    case SHAPE_HALF: return 16;
    default: return 8;
  }
}

// The shape of gemv where rows are read element by element in wide segments.  In double such loads are half as wide, so a
// thread has twice as many in flight, four rows instead of two (both products, us: 5003 x 3001 45.7 / 42.9, 3001 x 3001 29.4 /
// 26.1, 757600 x 141 353 / 291, 8001 x 8001 164 / 155; row product 20001 x 1001 with blocks of 64 KB as everywhere 27.2, of
// 128 KB 29.4).  Small matrices and few rows need the shorter blocks (2001 x 1001 11.4 / 12.5, 33 x 200001 25.9 / 26.5), and so
// does trmv (column sums n = 3581 26.4 / 27.2, row sums n = 1301 14.2 / 14.7).
constexpr double kWide4Elems = 4e6;
constexpr int64_t kWide4Rows = 1024;
template <typename T>
static int gemv_wide_shape(const L2Args<T>& a, int V) {
  return V == 1 && sizeof(T) == 8 && a.rows >= kWide4Rows && (double)a.rows * (double)a.cols >= kWide4Elems ? SHAPE_WIDE4 : SHAPE_WIDE;
}

// NARROW = false drops the two narrow shapes (kinds that never use them compile faster).
template <typename T, int V, class K, bool NARROW>
static int l2_launch(const Launch& l, const L2Args<T>& args, const L2Plan& plan, bool allow_direct) {
  if constexpr (V == 1 && sizeof(T) == 8 && K::TRI == TRI_FULL) {
    if (plan.shape == SHAPE_WIDE4)
      return l2_launch_shape<T, V, K, ShapeWide4>(l, args, plan.rows_per_cta, plan.ctiles_per_cta, allow_direct);
  }
  if (plan.shape == SHAPE_WIDE)
    return l2_launch_shape<T, V, K, ShapeWide>(l, args, plan.rows_per_cta, plan.ctiles_per_cta, allow_direct);
  if constexpr (NARROW) {
    if (plan.shape == SHAPE_HALF)
      return l2_launch_shape<T, V, K, ShapeHalf>(l, args, plan.rows_per_cta, plan.ctiles_per_cta, allow_direct);
    if (plan.shape == SHAPE_QUARTER)
      return l2_launch_shape<T, V, K, ShapeQuarter>(l, args, plan.rows_per_cta, plan.ctiles_per_cta, allow_direct);
  }
  return l2_launch_shape<T, V, K, ShapeMid>(l, args, plan.rows_per_cta, plan.ctiles_per_cta, allow_direct);
}

// Rows off 16-byte boundaries in shifted packs: where a row has more packs than the narrow shapes give it lanes and
// there is a whole step of rows.  In double, where element loads are only twice as many, they stay ahead for the
// kinds with one sum per element (gemv 8193 x 8191 175 us against 193, trmv n = 8191 95 against 112) and lose for
// symv (142 against 120).  Float: symv n = 8191 120 -> 72 us a pair, 11519 210 -> 115, trmv 8191 67 -> 58 with its
// copy, 11519 124 -> 100, gemv 8193 x 8191 108 -> 94.
// Row sums of short rows stay with element loads while the matrix is small (short_rows: up to which length).  Up to 1024
// elements a block covers the whole row then, and gemv needs no second pass: float 4000 x 512 6.4 us in shifted packs,
// 4.0 so, 1000 x 1000 5.0 / 4.5; with 707 columns 16 MB 6.5 / 6.1, 20 MB 6.6 / 7.0.  trmv: n = 256 5.3 / 4.0, 700 6.0 / 5.4,
// 900 5.7 / 6.0.
constexpr int kShortRowsGemv = 1024, kShortRowsTrmv = 768;
template <typename T>
static bool l2_shift(const L2Args<T>& a, bool sym, int short_rows) {
  constexpr int V = VecLen<T>::value;
  if (a.cols <= short_rows && (double)a.rows * (double)a.cols * sizeof(T) < 18e6) return false;
  return (sizeof(T) == 4 || sym) && !(aligned_to(a.a, 16) && a.lda % V == 0) && a.cols > 16 * V && a.rows >= ShapeMid::RB;
}

// Picks the pack width: 16-byte packs need a 16-byte aligned base and row stride.
template <typename T, class K, bool NARROW>
static int l2_dispatch(const Launch& l, const L2Args<T>& args, const L2Plan& plan, bool allow_direct) {
  constexpr int V = VecLen<T>::value;
  if (aligned_to(args.a, 16) && args.lda % V == 0) return l2_launch<T, V, K, NARROW>(l, args, plan, allow_direct);
  if (l2_shift(args, K::SYM, K::COLOUT ? 0 : K::TRI == TRI_FULL ? kShortRowsGemv : kShortRowsTrmv) && plan.shape == SHAPE_MID) {
    const int st = l2_launch_shape<T, V, K, ShapeMid, true>(l, args, plan.rows_per_cta, plan.ctiles_per_cta, allow_direct);
    if (st != B2_STATUS_WORKSPACE_TOO_SMALL) return st;
  }
  return l2_launch<T, 1, K, NARROW>(l, args, plan, allow_direct);
}

// Plans.  ROWOUT-only kinds: one row step per block, several column tiles per block so that a
// block streams about `tile_bytes`; the remaining column splits become partials.
template <typename T>
static L2Plan plan_rowout(const L2Args<T>& a, bool narrow_ok, int short_rows) {
  const bool shift = l2_shift(a, false, short_rows);
  const int V = (aligned_to(a.a, 16) && a.lda % VecLen<T>::value == 0) || shift ? VecLen<T>::value : 1;
  const int64_t nv = (a.cols + V - 1) / V;
  L2Plan p;
  // (shifted packs: short segments, 4 x values for 8 packs instead of 16)
  p.shape = nv >= 128 && !shift ? SHAPE_WIDE : (nv > 16 || !narrow_ok) ? SHAPE_MID : nv > 8 ? SHAPE_HALF : SHAPE_QUARTER;
  if (narrow_ok && p.shape == SHAPE_WIDE) p.shape = gemv_wide_shape(a, V);
  const int64_t tile_bytes = (int64_t)shape_rb(p.shape) * shape_packs_per_row(p.shape) * V * sizeof(T);
  int64_t cpc = knob(kKnobGemvNTileBytes) / tile_bytes;
  if (cpc < 1) cpc = 1;
  // (a row of up to 512 in one block, without a second pass: 12001 x 511 10.2 us, 11.5 in two, but 40001 x 301 19.7 and 19.0)
  if (p.shape == SHAPE_WIDE4 && a.cols <= 2 * cpc * shape_packs_per_row(p.shape)) cpc *= 2;
  // A matrix of a few long rows (at most 8 row steps) would get one partial per column split
  // and a finalize pass that adds thousands of them per row: there the splits are limited to
  // about eight resident blocks per SM in all.
  const int64_t nrs = (a.rows + shape_rb(p.shape) - 1) / shape_rb(p.shape);
  if (nrs <= 8) {
    const int64_t nct = (nv + shape_packs_per_row(p.shape) - 1) / shape_packs_per_row(p.shape);
    const int64_t want_ncs = std::max<int64_t>(1, (int64_t)sm_count() * 8 / nrs);
    cpc = std::max(cpc, (nct + want_ncs - 1) / want_ncs);
  }
  p.ctiles_per_cta = (int)cpc;
  p.tile_cols = shape_packs_per_row(p.shape) * V;
  p.rows_per_cta = shape_rb(p.shape);
  return p;
}
// COLOUT kinds: one column tile per block, tall row bands; the bands become partials.
template <typename T>
static L2Plan plan_colout(const L2Args<T>& a, bool narrow_ok, int64_t rows_per_cta) {
  const int V = (aligned_to(a.a, 16) && a.lda % VecLen<T>::value == 0) || l2_shift(a, false, 0) ? VecLen<T>::value : 1;
  const int64_t nv = (a.cols + V - 1) / V;
  L2Plan p;
  p.shape = (nv > 16 || !narrow_ok) ? SHAPE_MID : nv > 8 ? SHAPE_HALF : SHAPE_QUARTER;
  // element-wise rows (not 16-byte aligned): a 32-element column tile makes tiny blocks, take 128
  if (V == 1 && nv >= 128) p.shape = narrow_ok ? gemv_wide_shape(a, V) : SHAPE_WIDE;
  p.tile_cols = shape_packs_per_row(p.shape) * V;
  p.ctiles_per_cta = 1;
  if ((a.rows + rows_per_cta - 1) / rows_per_cta > 1024) rows_per_cta = (a.rows + 1023) / 1024;
  p.rows_per_cta = rows_per_cta;
  return p;
}

template <typename T>
static int scale_y(const Launch& l, T* y, int64_t incy, int64_t n, T beta) {
  if (beta == T(1) || n == 0) return B2_STATUS_OK;
  launch_chained(l2_scale_y<T>, dim3((unsigned)((n + kThreads - 1) / kThreads)), dim3(kThreads), 0, l.stream, vec_base(y, n, incy), incy, n, beta);
  return check_launch();
}

}  // namespace b2
