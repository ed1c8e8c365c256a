// trsv, cluster kernel: solve op(A) x = b in place (Section 6.2.2; same option space as trmv).
//
// The unknowns are cut into block rows of NB (64; 128 in float beyond the sizes of kShortRows), numbered in solve order.  The
// chain x_0 -> x_1 -> ... is the only sequential part; what it costs is the hand-over from one block
// row to the next, about 1 us through L2 and 0.2 us through the shared memory of a cluster.  So ONE
// cluster of kCS blocks walks the whole chain, and the other blocks of the grid stream the matrix:
//
//   solving block (rank c of the first cluster; block rows k = c, c + kCS, ...), block rows of 64
//     r   = b_k - far_k - u_W - ... - u_2      far_k from the streaming blocks, u_w = A(k, k-w) x(k-w)
//                                              from the cluster blocks that solved the rows before
//     x_k = inv(D_k) r - P_k x_(k-1)           P_k = inv(D_k) A(k, k-1), both in registers, one reduction
//     x_k stored straight into the shared memory of the block that owns row k + 1, and then
//     u   = A(k+w, k) x_k, w = 2 .. W          into those of the blocks that own rows k + w (the tiles through a
//                                              ring that one tiled copy per tile fills; off 16-byte boundaries by elements)
//     Between x_(k-1)'s arrival in row k and x_k's departure lie one register product and its reduction.  In block rows of 128 the
//     solving blocks' shared memory has no room to premultiply beside the near tiles: there u_1 travels, and two products and two
//     block barriers stand in the chain.
//   streaming block: 32-row strips of op(A), dealt out cyclically; at each step it multiplies the tiles
//     (strip, j), (strip, j + 1) of each of its strips that still needs them by x_j and x_(j+1) and keeps
//     the sums in registers.  Tile data does not depend on the solve, so a ring of 192 KB is always in
//     flight: every thread copies exactly the packs it later reads, so the ring needs no barrier.  A strip
//     of row k is complete after x(k-W-1); its sums are published W steps before the chain needs them,
//     which hides the two trips through L2.
//   The streaming blocks first invert the diagonal blocks of the rows beyond the first kCS and premultiply the tiles beside them
//   (off 16-byte boundaries those of the last rows, where it pays).
// Where P_k is not finite or has lost digits, where the workspace has no room for it and in rows 1 and 2, which the chain reaches
// first, row k's block keeps A(k, k-1) itself and multiplies twice.  An unknown that comes out infinite or NaN is formed once more in
// that way before it is sent on.
// The blocks of the first cluster start as solving ones -- they request and invert their diagonal blocks -- before they know
// their ticket; the others draw theirs a little later, and if the first cluster is late, one of them solves.
//
// Values cross blocks as tagged words (payload and ready flag in one store; the tag is unique per call
// in global memory, the row number in shared memory); consumers poll the data itself.  Every wait is
// bounded.  No co-residency is assumed: roles go by tickets drawn when a cluster starts, a streaming
// block only waits for the solving cluster (which drew the first ticket), and the solving cluster does
// the work of a streaming cluster that has not started yet itself, in the same order of additions.
//
// What bounds it: the chain, 0.6 us per block row of 64 in double and 0.5 in float (from x_k to the next: 0.2 us into the neighbour,
// 0.1 us of multiply-adds, 0.1 us of shuffles; from x_k by way of u_2 to x_(k+2) 0.55 us and as much again), 0.8 to 0.95 us per row of 128, after
// the start: 1.4 us until the diagonal block is there, 1.9 the inverse, 1 us of loads, and from row 3 on 2.1 the premultiplication
// (block rows of 128: 5.5 us the inverse).  From n = 11520 on in double, and off 16-byte boundaries from 8000 on, the streaming blocks
// (112 of them, the clusters leave 20 SMs idle), 5 TB/s.
// A copy and both solves, us, before the block rows of 64 in float, the premultiplied tiles, the tiled copies and the plain
// shared-memory polls / now: float n = 64 24.4 / 17.1, 192 29.9 / 19.0, 731 (unaligned) 45.9 / 31.9, 1000 45.1 / 34.6, 2048 53.7 / 50.8, 2322 (unaligned) 69.3 / 61.1,
// 4784 94.9 / 88.1, 11520 207.9 / 204.3, 13296 265 / 249; double 112 19.4 / 16.9, 608 32.7 / 28.7, 1024 42.2 / 36.7, 4224 118.8 / 104.2, 8512 229 / 206, 10417
// (unaligned) 479 / 474, 10752 291 / 271.  Slower: double off 16-byte boundaries, n = 4873 165.6 / 167.8, 8801 377 / 388; a first pass in double, whose matrix and code
// are not in L2, n = 300 39.1 / 42.4, 608 41 / 45, 1024 51.3 / 53.3, 1601 71.5 / 78 (but 2048 79.2 / 74.6; float 1000 55.2 / 49.5).
// Tried: clusters of 8 (column-type views 40 % slower in float: a block's pass over its near tiles takes
// longer than its turn), the near tiles on the receiving side (0.8 us more per row: the last of them then
// stands in the chain), one tile per ring slot (streaming alone 84 us instead of 51 us at n = 11520), the start's code run once on
// zeros ahead of the wait for the kernel before (no faster: it is not instruction fetches).
#include <algorithm>

#include "trsv_cluster.cuh"
#include "trsv_front.cuh"

namespace b2 {
namespace tc {

constexpr int kCS = 16;         // blocks per cluster (the opt-in size: 16 turns hide a row's preparation)
constexpr int kStrip = 32;      // rows of op(A) in a strip
constexpr int kStrips = 12;     // strips per streaming block at most
#ifdef B2_DEBUG_BOUNDS
constexpr bool kTma = false;  // (a TMA copy cannot be tested address by address)
#else
constexpr bool kTma = true;   // near tiles on 16-byte boundaries arrive as one tiled copy each
#endif
constexpr unsigned kNoTicket = 0xfffffffeu;  // not drawn yet
// Polls of the first cluster's ticket before another cluster draws one.  (A copy and two solves with 64 / without, us: float n = 1001
// 49.0 / 50.8, 3001 83.8 / 87.0, 11520 216 / 212, 16383 612 / 621, double 1024 42.5 / 44.2, 3001 105.8 / 100.5, 8192 225 / 220.)
constexpr int kHeadStart = 64;

template <typename T>
struct Args {
  const T* a;
  int64_t lda, n;
  T* x;  // base per vec_base()
  int64_t incx;
  u64* xbuf;         // [K * NB] published x
  u64* far;          // [K * NB] published row sums of the tiles left of the near window
  T* winv;           // [K - kCS][1 or 2][NB * NB] inverses of the diagonal blocks beyond the first kCS (and premultiplied tiles), as
                     // the solving blocks' threads hold them (Tile)
  u64* flags;        // [K] call tag once winv[k] is complete, below it whether there is a premultiplied tile
  int pm;            // tiles are premultiplied: 1 in the first kCS rows but the very first, 2 also beyond them from row pm_from on
  int pm_from;
  unsigned* ctl;
  int K;             // block rows
  int H;             // streaming blocks of the grid
  int W;             // rows behind the front whose tiles the solving cluster multiplies itself (at most G::W)
  int backward, unit;
  unsigned tag;
  u64 wait_limit;
  int* device_status;
  int debug_skip;
  int debug_late;  // test hook: polls for which the first cluster lets another one draw the first ticket
};

// Shared memory: one region that is the solving block's near-tile ring and inversion scratch or the
// streaming block's tile ring, then the small arrays.
template <class G>
struct Smem {
  using T = typename G::T;
  static constexpr int NB = G::NB, WPE = Words<T>::N;
  static constexpr size_t NEAR_TILE = (size_t)NB * NB * sizeof(T);
  static constexpr size_t NEAR_ELEMS = (size_t)G::NEAR * NB * NB;
  static constexpr bool WIDEN = sizeof(typename G::Wide) != sizeof(T);
  static constexpr size_t INV = sizeof(typename G::Wide) * Inv<G>::S_ELEMS * (G::PM ? 2 : 1);  // the inversion's scratch and the tile beside it
  static constexpr size_t SCRATCH = INV + (WIDEN ? sizeof(T) * Inv<G>::S_ELEMS * 2 : 0);       // and as they arrive, where they are widened
  static constexpr size_t SOLVE = G::NEAR * NEAR_TILE + SCRATCH;
  static constexpr size_t SLOT = 2 * (size_t)G::TP * kCT * 16;
  static constexpr size_t STREAM = G::DEPTH * SLOT;
  static constexpr size_t BIG = SOLVE > STREAM ? SOLVE : STREAM;
  static constexpr size_t RED = 2 * (size_t)kCW * NB * sizeof(T);  // cross-warp sums, two sets (also the inversion's Tm)
  static constexpr size_t TM = sizeof(typename G::Wide) * Inv<G>::TM_ELEMS;
  static constexpr size_t REDTM = RED > TM ? RED : TM;
  static constexpr size_t SLOTS = (size_t)G::W * NB * WPE * 8;  // sums of the rows 2 .. W behind; the first: of the row behind, or its x
  static constexpr size_t VECS = 4 * NB * sizeof(T);  // r, x of a row; two pairs of x blocks
  static constexpr size_t TOTAL = BIG + REDTM + SLOTS + VECS;
  // a streaming block inverts in the last slots of its ring, while the first ones fill
  static constexpr int FREE_SLOTS = (int)((STREAM - SCRATCH) / SLOT);
};

template <typename T>
struct Block {  // what both roles share
  T *big, *red, *rs, *xs;
  u64 *slots, *full;  // full: barriers of the near-tile ring (kTma)
  const CUtensorMap* map;
  Waiter wt;
  int tid, warp, lane;
  unsigned left, aborted;  // thread 0: blocks that had left before this one, the abort word then

  // This block looks at the ticket counter no more.  The answers are awaited at the kernel's end only.  (Asked for there, one
  // after the other behind the last row, they made a solve 0.5 us longer.)
  __device__ __forceinline__ void leave(unsigned* ctl) {
    look_and_count_if(tid == 0, ctl + kCtlTrsvAbort, ctl + kCtlTrsvDone, aborted, left);
  }
};

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
// offset in the block's dynamic shared memory
__device__ __forceinline__ unsigned smem_off(const void* p) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  return smem_addr(p) - smem_addr(smem_raw);
}

// Memory index of the block row at position k of the solve order.
template <typename T>
__device__ __forceinline__ int mem_block(const Args<T>& p, int k) { return p.backward ? p.K - 1 - k : k; }
template <int NB, typename T>
__device__ __forceinline__ int block_len(const Args<T>& p, int I) { return (int)min((int64_t)NB, p.n - (int64_t)I * NB); }

// Whether the cluster that holds streaming block h has started (its ticket has been drawn).
template <typename T>
__device__ __forceinline__ bool has_started(const Args<T>& p, int h) {
  return ld_flag(p.ctl + kCtlTrsvTicket) > (unsigned)(1 + h / kCS);
}

// ---- a strip's tile ------------------------------------------------------------------------------------
// Sums of a thread.  Row-type views (op(A)'s rows contiguous): warp w holds rows 4w .. 4w + 3 of the
// strip, a lane V columns of each (of every second one, where a row has only 16 packs), one sum per row.  Column-type views: the warp's lanes run along the
// strip (contiguous in memory), over NB / 8 columns of the tile; V sums per lane, one per row of op(A).
template <class G, bool COLTYPE>
struct Strip {
  using T = typename G::T;
  static constexpr int NB = G::NB, V = G::V, TP = G::TP;
  static constexpr int NA = COLTYPE ? V : TP;
  static constexpr int LPR = kStrip / V, GR = 32 / LPR;  // column-type: lanes along the strip, stored rows per instruction
  static constexpr int RL = NB / V, RG = 32 / RL;        // row-type: lanes along a row, rows per instruction
  static_assert(kCW * TP * GR == NB && kCW * TP * RG == kStrip, "every element of the tile exactly once");

  // the thread's first element of the tile: row of op(A) and column
  __device__ __forceinline__ static int row0(int warp, int lane) { return COLTYPE ? (lane % LPR) * V : warp * TP * RG + lane / RL; }
  __device__ __forceinline__ static int col0(int warp, int lane) { return COLTYPE ? warp * (NB / kCW) + lane / LPR : lane % RL * V; }

  // address and number of existing elements of pack q of this thread
  __device__ __forceinline__ static const T* pack_ptr(const Args<T>& p, int I, int sub, int J, int warp, int lane, int q, int* valid) {
    const int i = sub * kStrip + row0(warp, lane) + (COLTYPE ? 0 : RG * q), j = col0(warp, lane) + (COLTYPE ? GR * q : 0);
    const int rl = (COLTYPE ? block_len<NB>(p, J) - j : block_len<NB>(p, I) - i), cl = (COLTYPE ? block_len<NB>(p, I) - i : block_len<NB>(p, J) - j);
    *valid = rl > 0 ? (cl < 0 ? 0 : cl > V ? V : cl) : 0;
    const int64_t r = (int64_t)(COLTYPE ? J : I) * NB + (COLTYPE ? j : i), c = (int64_t)(COLTYPE ? I : J) * NB + (COLTYPE ? i : j);
    return p.a + r * p.lda + c;
  }
  // this thread's values of x for every tile of a block column
  static constexpr int NX = COLTYPE ? TP : V;
  __device__ __forceinline__ static void load_x(T (&x)[NX], const T* xv, int warp, int lane) {
    if constexpr (!COLTYPE) {
      ld_pack(xv + col0(warp, lane), x);
    } else {
#pragma unroll
      for (int q = 0; q < TP; ++q) x[q] = xv[col0(warp, lane) + GR * q];
    }
  }
  __device__ __forceinline__ static void add(T (&acc)[NA], const Pack<T, V> (&m)[TP], const T (&x)[NX]) {
#pragma unroll
    for (int q = 0; q < TP; ++q)
#pragma unroll
      for (int e = 0; e < V; ++e) {
        if (!COLTYPE) acc[q] = m[q].v[e] * x[e] + acc[q];
        else acc[e] = m[q].v[e] * x[q] + acc[e];
      }
  }
};

// Complete row sums of a strip from its threads' sums -> far words of block row k.  All threads.
template <class G, bool COLTYPE>
__device__ __forceinline__ typename G::T strip_rows(const typename G::T (&sum)[Strip<G, COLTYPE>::NA], typename G::T* red, int warp, int lane, int* row) {
  using ST = Strip<G, COLTYPE>;
  using T = typename G::T;
  if constexpr (!COLTYPE) {  // the first lane of every few gets a row
    T v[ST::TP];
#pragma unroll
    for (int q = 0; q < ST::TP; ++q) v[q] = sum[q];
    const T s = multi_group_sum<ST::RL, ST::TP>(v, lane);
    constexpr int LPV = ST::RL / ST::TP;
    *row = lane % LPV == 0 ? ST::row0(warp, lane) + ST::RG * (lane % ST::RL / LPV) : -1;
    return s;
  } else {  // warp 0 gets the rows
    Pack<T, ST::V> pk;
#pragma unroll
    for (int e = 0; e < ST::V; ++e) pk.v[e] = cross_group_sum<ST::LPR>(sum[e]);
    if (lane < ST::LPR) *reinterpret_cast<Pack<T, ST::V>*>(red + warp * kStrip + lane * ST::V) = pk;
    bar_block();
    T s = T(0);
    if (warp == 0) {
#pragma unroll
      for (int w = 0; w < kCW; ++w) s += red[w * kStrip + lane];
    }
    *row = warp == 0 ? lane : -1;
    return s;
  }
}

// ---- a tile in the registers of a solving block ----------------------------------------------------------
// A 16 x 16 thread grid: thread (rg, cg) holds rows RS rg .. RS rg + RS - 1 and of each the CP packs V cg + e, H + V cg + e, ...:
// one or two 16-byte shared-memory loads fetch its part of a vector and the row sums run over 16 lanes.  (One row per four threads
// needs eight loads per thread, and even a broadcast load occupies the load path for its 512 bytes of results: 0.55 us a product.)
template <class G>
struct Tile {
  using T = typename G::T;
  static constexpr int NB = G::NB, V = G::V, RS = NB / 16, H = 16 * V, CP = NB / H, NPK = RS * CP;
  using P = Pack<T, V>;
  // a pack of T or of wider elements
  template <typename U>
  __device__ __forceinline__ static P pack_of(const U* q) {
    if constexpr (sizeof(U) == sizeof(T)) {
      return *reinterpret_cast<const P*>(q);
    } else {
      P r;
#pragma unroll
      for (int e = 0; e < V; e += 2) {
        const double2 d = *reinterpret_cast<const double2*>(q + e);
        r.v[e] = (T)d.x, r.v[e + 1] = (T)d.y;
      }
      return r;
    }
  }
  // rows at src
  template <typename U>
  __device__ __forceinline__ static void from_rows(P (&t)[NPK], const U* src, int pitch, int tid) {
    const int rg = tid >> 4, cg = tid & 15;
#pragma unroll
    for (int m = 0; m < NPK; ++m) t[m] = pack_of(src + (rg * RS + m / CP) * pitch + (m % CP) * H + cg * V);
  }
  // columns at src; ld: how a pack is loaded
  template <typename U, class Load>
  __device__ __forceinline__ static void from_columns(P (&t)[NPK], const U* src, int64_t pitch, int tid, Load ld) {
    const int rg = tid >> 4, cg = tid & 15;
#pragma unroll
    for (int h = 0; h < CP; ++h)
#pragma unroll
      for (int e = 0; e < V; ++e)
#pragma unroll
        for (int a = 0; a < RS; a += V) {
          const P pk = ld(src + (h * H + cg * V + e) * pitch + rg * RS + a);
#pragma unroll
          for (int u = 0; u < V; ++u) t[(a + u) * CP + h].v[e] = pk.v[u];
        }
  }
  // The inverse in S, or its transpose; that with a thread's columns 16 apart (cg, cg + 16, ...), so that the rows of S that
  // neighbouring lanes read lie in different banks (apart as in the other layout, an inverse took 1900 cycles instead of 600).
  __device__ __forceinline__ static void inverse(P (&t)[NPK], const typename G::Wide* S, bool transposed, int tid) {
    if (!transposed) {
      from_rows(t, S, Inv<G>::SP, tid);
    } else {
      const typename G::Wide* q = S + (tid & 15) * Inv<G>::SP + (tid >> 4) * RS;
#pragma unroll
      for (int c = 0; c < CP * V; ++c)
#pragma unroll
        for (int a = 0; a < RS; a += V) {
          const P pk = pack_of(q + c * 16 * Inv<G>::SP + a);
#pragma unroll
          for (int u = 0; u < V; ++u) t[(a + u) * CP + c / V].v[c % V] = pk.v[u];
        }
    }
  }
  // this thread's part of the vector that the inverse is multiplied by
  __device__ __forceinline__ static void load_r(P (&x)[CP], const T* vec, bool transposed, int tid) {
    if (!transposed) {
      load_x(x, vec, tid);
    } else {
#pragma unroll
      for (int c = 0; c < CP * V; ++c) x[c / V].v[c % V] = vec[(tid & 15) + c * 16];
    }
  }
  // as the threads hold it, in global memory
  __device__ __forceinline__ static void store(const P (&t)[NPK], T* dst, int tid) {
#pragma unroll
    for (int m = 0; m < NPK; ++m) *reinterpret_cast<P*>(dst + ((size_t)m * kCT + tid) * V) = t[m];
  }
  __device__ __forceinline__ static void load(P (&t)[NPK], const T* src, int tid) {
#pragma unroll
    for (int m = 0; m < NPK; ++m) t[m] = ld_cg_if<T, V>(src + ((size_t)m * kCT + tid) * V, true);
  }
  // this thread's part of a vector
  __device__ __forceinline__ static void load_x(P (&x)[CP], const T* vec, int tid) {
#pragma unroll
    for (int h = 0; h < CP; ++h) x[h] = *reinterpret_cast<const P*>(vec + h * H + (tid & 15) * V);
  }
  // The row whose sum a thread ends up with (the first of every few lanes: its owner).
  __device__ __forceinline__ static int row(int tid) { return (tid >> 4) * RS + (tid & 15) / (16 / RS); }
  // Where the words of element i of x_(k-1) lie in a solving block's first slots: what neighbouring lanes read side by side.
  __device__ __forceinline__ static unsigned x_word(unsigned slots, int i) {
    constexpr int WPE = Words<T>::N;
    return slots + (unsigned)(((i / H * 2 + i % V * WPE / 2) * 16 + i % H / V) * 16 + i % V * WPE % 2 * 8);
  }
  // Sums of a thread's rows, in float of even and odd columns side by side (packed multiply-adds).
  struct Sums {
    typename std::conditional<sizeof(T) == 4, u64, T>::type v[RS];
  };
  // tile * x
  __device__ __forceinline__ static void multiply(Sums& s, const P (&t)[NPK], const P (&x)[CP]) {
#pragma unroll
    for (int h = 0; h < CP; ++h) {
      if constexpr (sizeof(T) == 4) {
        const ulonglong2 x2 = *reinterpret_cast<const ulonglong2*>(&x[h]);
#pragma unroll
        for (int a = 0; a < RS; ++a) {
          const ulonglong2 m2 = *reinterpret_cast<const ulonglong2*>(&t[a * CP + h]);
          s.v[a] = fma2(m2.x, x2.x, h == 0 ? 0ull : s.v[a]);
          s.v[a] = fma2(m2.y, x2.y, s.v[a]);
        }
      } else {
#pragma unroll
        for (int e = 0; e < V; ++e)
#pragma unroll
          for (int a = 0; a < RS; ++a) s.v[a] = h == 0 && e == 0 ? t[a * CP].v[0] * x[0].v[0] : t[a * CP + h].v[e] * x[h].v[e] + s.v[a];
      }
    }
  }
  __device__ __forceinline__ static T of(u64 pair) { return __uint_as_float((unsigned)pair) + __uint_as_float((unsigned)(pair >> 32)); }
  __device__ __forceinline__ static T of(double sum) { return sum; }
  // The whole sum of the row that this lane ends up with: row rg RS + cg / (16 / RS).  Of two products: each is added up by itself
  // first, so that the smaller one's additions are rounded at its own size.
  __device__ __forceinline__ static T reduce(const Sums& s, int lane) {
    T acc[RS];
#pragma unroll
    for (int a = 0; a < RS; ++a) acc[a] = of(s.v[a]);
    return multi_group_sum<16, RS>(acc, lane);
  }
  __device__ __forceinline__ static T reduce(const Sums& s, const Sums& s2, int lane) {
    T acc[RS];
#pragma unroll
    for (int a = 0; a < RS; ++a) acc[a] = of(s.v[a]) + of(s2.v[a]);
    return multi_group_sum<16, RS>(acc, lane);
  }
  __device__ __forceinline__ static T product(const P (&t)[NPK], const P (&x)[CP], int lane) {
    Sums s;
    multiply(s, t, x);
    return reduce(s, lane);
  }
  // The same of the inverse and load_r's vector, without the zeros on the other side of the diagonal: an infinite or NaN element of
  // the vector takes no unknowns along that do not depend on it.
  __device__ __forceinline__ static T triangle(const P (&t)[NPK], const P (&x)[CP], bool transposed, int tid) {
    const int rg = tid >> 4, cg = tid & 15;
    T acc[RS];
#pragma unroll
    for (int a = 0; a < RS; ++a) {
      acc[a] = T(0);
#pragma unroll
      for (int c = 0; c < CP * V; ++c) {
        const int i = rg * RS + a, j = transposed ? c * 16 + cg : c / V * H + cg * V + c % V;
        if (transposed ? j >= i : j <= i) acc[a] = t[a * CP + c / V].v[c % V] * x[c / V].v[c % V] + acc[a];
      }
    }
    return multi_group_sum<16, RS>(acc, tid & 31);
  }
};

// acc[s] += tiles * x with s known at run time (the sums stay in registers); both: the second tile counts;
// done: the sums, when `last`.
template <class ST, int I, typename T>
__device__ __forceinline__ void add_to(T (&acc)[kStrips][ST::NA], int s, const Pack<T, ST::V> (&m)[2][ST::TP], const T (&x)[2][ST::NX], bool both,
                                       bool last, T (&done)[ST::NA]) {
  if (s == I) {
    ST::add(acc[I], m[0], x[0]);
    if (both) ST::add(acc[I], m[1], x[1]);
    if (last) {
#pragma unroll
      for (int e = 0; e < ST::NA; ++e) done[e] = acc[I][e];
    }
  } else if constexpr (I + 1 < kStrips) {
    add_to<ST, I + 1>(acc, s, m, x, both, last, done);
  }
}

// Shared memory of the inversion: S, the tile beside it, and both as they arrive (the same places where nothing is widened).
template <class G>
struct Scratchpad {
  using T = typename G::T;
  using U = typename G::Wide;
  U *S, *N;
  T *s, *n;
  __device__ __forceinline__ explicit Scratchpad(void* at) {
    S = reinterpret_cast<U*>(at), N = S + Inv<G>::S_ELEMS;
    if constexpr (Smem<G>::WIDEN) s = reinterpret_cast<T*>(reinterpret_cast<unsigned char*>(at) + Smem<G>::INV), n = s + Inv<G>::S_ELEMS;
    else s = S, n = N;
  }
  // what has arrived (both: the tile as well) -> S, N.  All threads; ends without a barrier.
  __device__ __forceinline__ void arrived(bool both, int tid) const {
    if constexpr (Smem<G>::WIDEN) widen<G>(S, s, (both ? 2 : 1) * Inv<G>::S_ELEMS, tid);
  }
};

// Diagonal block I once more, from the matrix (cold path; all copies of this thread that are in flight are waited for).
template <class G, bool COLTYPE, bool AL>
__device__ __noinline__ void invert_again(const Args<typename G::T>& p, unsigned s_off, int I, int tid) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const Scratchpad<G> pad(smem_raw + s_off);
  Diag<G, COLTYPE, AL>::stage(p.a, p.lda, p.n, I, p.backward, pad.s, tid);
  cp_async_wait<0>();
  pad.arrived(false, tid);
  bar_block();
  invert_rows<G>(pad.S, p.unit, block_len<G::NB>(p, I), tid);
}
// Its inverse by a solving block for which no other one forms it (cold path, as above).
template <class G, bool COLTYPE, bool AL>
__device__ __noinline__ void form_inverse(const Args<typename G::T>& p, unsigned s_off, unsigned tm_off, int I, int tid) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const Scratchpad<G> pad(smem_raw + s_off);
  Diag<G, COLTYPE, AL>::stage(p.a, p.lda, p.n, I, p.backward, pad.s, tid);
  cp_async_wait<0>();
  pad.arrived(false, tid);
  bar_block();
  if (invert_block<G>(s_off, tm_off, p.unit, block_len<G::NB>(p, I), tid)) invert_again<G, COLTYPE, AL>(p, s_off, I, tid);
}
// Tile (I, J) of op(A) as it is stored, beside it (cold path, as above).
template <class G, bool COLTYPE, bool AL>
__device__ __noinline__ void fetch_tile(const Args<typename G::T>& p, unsigned s_off, int I, int J, int tid) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const Scratchpad<G> pad(smem_raw + s_off);
  bar_block();
  stage_tile<G, COLTYPE, AL>(p.a, p.lda, I, J, block_len<G::NB>(p, I), block_len<G::NB>(p, J), pad.n, tid);
  cp_async_commit();
  cp_async_wait<0>();
  bar_block();
}

// inv r and P x may be beyond the type where inv (r - A x) is not, and an infinite element of r must not take those before it along:
// the unknown that this lane ends up with (Tile) once more, as inv(D_k) (r - A(k, k-1) x_(k-1)) without the zeros of the inverse, by
// its warp alone, and where it is to go, if `out`.  Where x_(k-1) is not finite it stays what it is, x (what follows is not finite
// either).  Cold path; offsets in shared memory, own: of the warp; inverse: in global memory, or null: in S.
template <class G, bool COLTYPE>
__device__ __noinline__ void solve_apart(const Args<typename G::T>& p, const typename G::T* inverse, unsigned s_off, unsigned slots, unsigned r_off,
                                         unsigned own_off, int k, int tid, bool transposed, bool out, typename G::T x) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  using T = typename G::T;
  using TL = Tile<G>;
  constexpr int NB = G::NB, WPE = Words<T>::N;
  T* const r = reinterpret_cast<T*>(smem_raw + r_off);
  T* const own = reinterpret_cast<T*>(smem_raw + own_off);
  const int I = mem_block(p, k), J = mem_block(p, max(k - 1, 0)), li = block_len<NB>(p, I), lj = k > 0 ? block_len<NB>(p, J) : 0, lane = tid & 31;
  u64 wd[WPE];
  double before[NB / 32];
  bool finite = true;
#pragma unroll
  for (int c = 0; c < NB / 32; ++c) {
    ld_slot(TL::x_word(slots, lane + 32 * c), wd);
    before[c] = k > 0 ? (double)decode(wd, T(0)) : 0.;
    finite = finite && isfinite(before[c]);
  }
  if (__all_sync(0xffffffffu, finite)) {
#pragma unroll 8
    for (int i = 0; i < NB; ++i) {
      double s = 0.;
#pragma unroll
      for (int c = 0; c < NB / 32; ++c) {
        const int j = lane + 32 * c;
        const int64_t m = (int64_t)I * NB + i, q = (int64_t)J * NB + j;
        if (i < li && j < lj) s += (double)__ldg(p.a + (COLTYPE ? q * p.lda + m : m * p.lda + q)) * before[c];
      }
      s = cross_group_sum<1>(s);
      if (lane == 0) own[i] = (T)((double)r[i] - s);
    }
    __syncwarp();
    typename TL::P inv[TL::NPK], v[TL::CP];
    if (inverse) TL::load(inv, inverse, tid);
    else TL::inverse(inv, reinterpret_cast<const typename G::Wide*>(smem_raw + s_off), transposed, tid);
    TL::load_r(v, own, transposed, tid);
    x = TL::triangle(inv, v, transposed, tid);
  }
  const int row = TL::row(tid);
  encode(x, (unsigned)k + 2u, wd);
  st_slot_if(out && k + 1 < p.K, map_remote(TL::x_word(slots, row), (unsigned)((k + 1) % kCS)), wd);
  if (out) r[NB + row] = x;  // (x of the row)
  encode(x, p.tag, wd);
  st_gpu_if(out, p.xbuf + ((int64_t)k * NB + row) * WPE, wd);
  st_val_if(out && row < li, p.x + ((int64_t)I * NB + min(row, li - 1)) * p.incx, x);
  bar_block();
}

// ---- streaming block -----------------------------------------------------------------------------------
template <class G, bool COLTYPE, bool AL>
__device__ __forceinline__ void stream_block(const Args<typename G::T>& p, Block<typename G::T>& b, int h) {
  using T = typename G::T;
  using ST = Strip<G, COLTYPE>;
  constexpr int NB = G::NB, V = G::V, WPE = Words<T>::N, SPB = NB / kStrip;  // strips per block row
  constexpr int TP = G::TP, kDepth = G::DEPTH;
  const int W = p.W;
  // strip s of this block is strip q0 + h + s * H of the matrix; it needs the tiles j = 0 .. k - W - 1
  const int q0 = (W + 1) * SPB + h, nstrips = p.K * SPB, H = p.H;
  const int S = q0 >= nstrips ? 0 : min(kStrips, (nstrips - q0 + H - 1) / H);
  const int jmax = S > 0 ? (q0 + (S - 1) * H) / SPB - W - 1 : -1;
  const int ragged = (int)(p.n % NB) != 0 ? p.K - 1 : -1;  // memory index of the block that is not full

  T acc[kStrips][ST::NA];
#pragma unroll
  for (int s = 0; s < kStrips; ++s)
#pragma unroll
    for (int e = 0; e < ST::NA; ++e) acc[s][e] = T(0);

  // what the loop needs to know of the strips, once per block: last block column, offset of the first element
  __shared__ int s_last[kStrips];
  __shared__ int64_t s_base[kStrips];
  if (b.tid < S) {
    const int q = q0 + b.tid * H;
    s_last[b.tid] = q / SPB - W - 1;
    s_base[b.tid] = ((int64_t)mem_block(p, q / SPB) * NB + q % SPB * kStrip) * (COLTYPE ? 1 : p.lda);
  }
  bar_block();

  // producer: the sequence (j, s), j = 0, 2, ..., s over the strips that still need tile j, up to kDepth slots ahead
  int pj = 0, plo = 0, ps = 0, pslot = 0;
  const T* const at = p.a + (COLTYPE ? ST::col0(b.warp, b.lane) * p.lda + ST::row0(b.warp, b.lane) : ST::row0(b.warp, b.lane) * p.lda + ST::col0(b.warp, b.lane));
  const T* const uat = p.a + (COLTYPE ? ST::col0(b.warp, 0) : ST::row0(b.warp, 0)) * p.lda + b.lane;
  const int64_t step_a = (COLTYPE ? ST::GR : ST::RG) * p.lda;
  auto off_e = [&](int e) { return COLTYPE ? e * p.lda : e * 32 / NB * p.lda + e * 32 % NB; };  // (copy_warp)
  const int64_t jstep = (COLTYPE ? p.lda : 1) * (p.backward ? -NB : NB);  // from a block column to the next in solve order
  const int64_t j0off = (COLTYPE ? p.lda : 1) * (int64_t)mem_block(p, 0) * NB;
  auto produce = [&]() {
    if (pj <= jmax) {
      T* dst = b.big + ((size_t)(pslot * 2 * TP) * kCT + b.tid) * V;
      const bool both = pj < s_last[ps];
      const bool whole = ragged < 0 || (p.backward ? pj > 0 : (q0 + ps * H) / SPB != ragged);
      if (whole) {
        const int64_t tile = s_base[ps] + j0off + pj * jstep;
        if constexpr (AL) {
          const T* src = at + tile;
#pragma unroll
          for (int r = 0; r < TP; ++r) cp_async16_full(dst + (size_t)r * kCT * V, src + r * step_a);
          if (both) {
#pragma unroll
            for (int r = 0; r < TP; ++r) cp_async16_full(dst + (size_t)(TP + r) * kCT * V, src + jstep + r * step_a);
          }
        } else {
          const T* src = uat + tile;
          dst -= b.lane * (V - 1);
#pragma unroll
          for (int r = 0; r < TP; ++r) copy_warp(dst + (size_t)r * kCT * V, src + r * step_a, off_e);
          if (both) {
#pragma unroll
            for (int r = 0; r < TP; ++r) copy_warp(dst + (size_t)(TP + r) * kCT * V, src + jstep + r * step_a, off_e);
          }
        }
      } else {
        const int q = q0 + ps * H;
#pragma unroll 1
        for (int r = 0; r < (both ? 2 : 1) * TP; ++r) {
          int valid;
          const T* src = ST::pack_ptr(p, mem_block(p, q / SPB), q % SPB, mem_block(p, pj + r / TP), b.warp, b.lane, r % TP, &valid);
          copy_pack<T, AL>(dst + (size_t)r * kCT * V, src, valid, p.a);
        }
      }
      if (++ps == S) {
        pj += 2;
        while (plo < S - 1 && s_last[plo] < pj) ++plo;
        ps = plo;
      }
    }
    cp_async_commit();
    pslot = pslot + 1 == kDepth ? 0 : pslot + 1;
  };
  // Diagonal blocks, dealt out from the last block on (the first ones have the most urgent strips), and in
  // the meantime the first tiles.
  int filled = 0;
#pragma unroll 1
  for (int k = kCS + p.H - 1 - h; k < p.K; k += p.H) {
    const Scratchpad<G> pad(reinterpret_cast<unsigned char*>(b.big) + Smem<G>::STREAM - Smem<G>::SCRATCH);
    const unsigned at = smem_off(pad.S);
    const int I = mem_block(p, k), J = mem_block(p, k - 1);
    const bool room = G::PM && p.pm > 1, pm = room && k >= p.pm_from;
    if constexpr (G::PM) {
      if (pm) stage_tile<G, COLTYPE, AL>(p.a, p.lda, I, J, block_len<NB>(p, I), block_len<NB>(p, J), pad.n, b.tid);
    }
    Diag<G, COLTYPE, AL>::stage(p.a, p.lda, p.n, I, p.backward, pad.s, b.tid);
    if (filled == 0) {
#pragma unroll 1
      for (; filled < Smem<G>::FREE_SLOTS; ++filled) produce();
      cp_async_wait<Smem<G>::FREE_SLOTS>();
    } else {
      cp_async_wait<0>();
    }
    pad.arrived(pm, b.tid);
    bar_block();
    if (invert_block<G>(at, smem_off(b.red), p.unit, block_len<NB>(p, I), b.tid)) invert_again<G, COLTYPE, AL>(p, at, I, b.tid);
    const bool transposed = Diag<G, COLTYPE, AL>::transposed(p.backward);
    T* dst = p.winv + (int64_t)(k - kCS) * NB * NB * (room ? 2 : 1);
    typename Tile<G>::P t[Tile<G>::NPK];
    Tile<G>::inverse(t, pad.S, transposed, b.tid);
    Tile<G>::store(t, dst, b.tid);
    unsigned have = 0;
    if constexpr (G::PM) {
      if (pm && !premultiply<G, COLTYPE>(at, smem_off(pad.N), transposed, block_len<NB>(p, I), block_len<NB>(p, J), b.tid)) {
        have = 1;
        Tile<G>::from_rows(t, pad.N, Inv<G>::SP, b.tid);
        Tile<G>::store(t, dst + NB * NB, b.tid);
      }
    }
    __threadfence();
    bar_block();
    if (b.tid == 0) st_flag(p.flags + k, (u64)p.tag << 32 | have);
  }
#pragma unroll 1
  for (; filled < kDepth - 1; ++filled) produce();

  // x_j and x_(j+1): one word per thread (a block's x is 128 words, 64 in the small float blocks), loaded a step ahead; into
  // one of two shared-memory buffers, then one block barrier per step.  (x_(j+1) is there long before the
  // row that a strip with last tile j belongs to is due.)
  static_assert(2 * NB * WPE <= kCT, "one word per thread at most");
  const bool has_word = 2 * NB * WPE == kCT || b.tid < 2 * NB * WPE;
  const u64* xsrc = p.xbuf + b.tid;
  u64 xw[1];
  if (jmax >= 0 && has_word) ld_gpu(xsrc, xw);
  int slot = 0, lo = 0, par = 0;
  auto finish = [&](int q, const T (&sum)[ST::NA]) {  // strip q is complete
    int row;
    const T v = strip_rows<G, COLTYPE>(sum, b.red + par * (kCW * kStrip), b.warp, b.lane, &row);
    par ^= 1;
    u64 wd[WPE];
    encode(v, p.tag, wd);
    st_gpu_if(row >= 0 && !*b.wt.dead, p.far + ((int64_t)(q / SPB) * NB + (q % SPB) * kStrip + max(row, 0)) * WPE, wd);
  };
#pragma unroll 1
  for (int j = 0; j <= jmax; j += 2) {
    T* xv = b.rs + (j & 2) * NB;  // (xs: four blocks)
    auto receive = [&]() {
      if (!has_word) return;
      while (!tagged(xw, p.tag)) {
        if (!b.wt.again()) break;
        ld_gpu(xsrc, xw);
      }
      reinterpret_cast<unsigned*>(xv)[b.tid] = (unsigned)xw[0];  // (a double is its two payload halves, low first)
      xsrc += 2 * NB * WPE;
      if (j + 2 <= jmax) ld_gpu(xsrc, xw);
    };
    while (lo < S - 1 && s_last[lo] < j) ++lo;
    // A strip that ends with tile j goes first and without x_(j+1), which the chain has one row later: its sums are due
    // W rows after x_j.  (With both awaited, every second row of the chain waited for them: a pair of solves of n = 11520
    // took 2 % longer.  In double the slack is longer, off 16-byte boundaries the strips take longer, and the second barrier
    // costs more: double n = 9008 2 %, float n = 8191 3 % longer with it.)
    const bool alone = sizeof(T) == 4 && NB == 128 && AL && s_last[lo] == j;
    const bool second = b.tid >= NB * WPE;  // this thread's word belongs to x_(j+1)
    if (!(alone && second)) receive();
    bar_block();
    T x[2][ST::NX];
    ST::load_x(x[0], xv, b.warp, b.lane);
    if (!alone) ST::load_x(x[1], xv + NB, b.warp, b.lane);
#pragma unroll 1
    for (int s = lo; s < S; ++s) {
      if (alone && s == lo + 1) {
        if (second) receive();
        bar_block();
        ST::load_x(x[1], xv + NB, b.warp, b.lane);
      }
      if (!AL) __syncwarp();  // (a warp's copies are spread over its lanes: the slot's readers are done)
      produce();
      const int last_j = s_last[s];
      const T* src = b.big + ((size_t)(slot * 2 * TP) * kCT + b.tid) * V;
      slot = slot + 1 == kDepth ? 0 : slot + 1;
      cp_async_wait<kDepth - 1>();
      if (!AL) __syncwarp();
      Pack<T, V> m[2][TP];
#pragma unroll
      for (int r = 0; r < 2 * TP; ++r)
        m[r / TP][r % TP] = *reinterpret_cast<const Pack<T, V>*>(src + (size_t)r * kCT * V);
      T done[ST::NA];
      add_to<ST, 0>(acc, s, m, x, j < last_j, last_j - j <= 1, done);
      if (last_j - j <= 1) finish(q0 + s * H, done);
    }
  }
  cp_async_wait<0>();
}

// Row sums of a strip that no running block will deliver, by one warp of the solving block (lane i:
// row i of the strip), with the additions of a streaming block in the same order.
template <class G, bool COLTYPE>
__device__ __noinline__ typename G::T slow_strip(const Args<typename G::T>& p, int k, int sub, int jend, Waiter wt, int lane) {
  using T = typename G::T;
  using ST = Strip<G, COLTYPE>;
  constexpr int NB = G::NB, V = G::V, WPE = Words<T>::N, TP = G::TP;
  const int I = mem_block(p, k);
  T out = T(0);
  for (int w = 0; w < kCW; ++w) {
    T acc[ST::NA];
#pragma unroll
    for (int e = 0; e < ST::NA; ++e) acc[e] = T(0);
    for (int j = 0; j < jend; ++j) {
      const int J = mem_block(p, j);
      auto x_at = [&](int i) {
        u64 wd[WPE];
        const u64* q = p.xbuf + ((int64_t)j * NB + i) * WPE;
        ld_gpu(q, wd);
        while (!tagged(wd, p.tag) && wt.again()) ld_gpu(q, wd);
        return decode(wd, T(0));
      };
#pragma unroll
      for (int r = 0; r < TP; ++r) {
        int valid;
        const T* src = ST::pack_ptr(p, I, sub, J, w, lane, r, &valid);
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const T m = e < valid ? __ldg(src + e) : T(0);
          if (!COLTYPE) acc[r] = m * x_at(ST::col0(w, lane) + e) + acc[r];
          else acc[e] = m * x_at(ST::col0(w, lane) + ST::GR * r) + acc[e];
        }
      }
    }
    __syncwarp();
    if constexpr (!COLTYPE) {
      const T s = multi_group_sum<ST::RL, TP>(acc, lane);
      const int q = lane % (TP * ST::RG);  // row 4 w + q of the strip is group q % RG's sum q / RG
      const T mine = __shfl_sync(0xffffffffu, s, q % ST::RG * ST::RL + q / ST::RG * (ST::RL / TP));
      if (lane / (TP * ST::RG) == w) out = mine;
    } else {
#pragma unroll
      for (int e = 0; e < V; ++e) {
        const T s = cross_group_sum<ST::LPR>(acc[e]);  // of row V * (lane % LPR) + e
        const T mine = __shfl_sync(0xffffffffu, s, lane / V);
        if (lane % V == e) out += mine;
      }
    }
  }
  return out;
}

// Draws the ticket of a cluster and hands it to its blocks.  One thread of the cluster's first block.
template <typename T>
__device__ __forceinline__ void draw_ticket(const Args<T>& p, unsigned* ticket, bool early) {
  unsigned t = 0xffffffffu;
  // The first cluster, whose blocks start as solving ones, is let go first; if it has not started after a while, another
  // one solves.
  const int polls = early ? p.debug_late : kHeadStart;
  for (int i = 0; i < polls && ld_flag(p.ctl + kCtlTrsvTicket) == 0u; ++i) {}
  // (abort word up: left by an earlier timed-out call on a workspace that was not reset, or raised
  // meanwhile: nothing is solved, and the caller must be able to see that)
  if (ld_flag(p.ctl + kCtlTrsvAbort) == 0u) t = atomicAdd(p.ctl + kCtlTrsvTicket, 1u);
  else if (p.device_status) atomicExch(p.device_status, (int)B2_STATUS_TIMEOUT);
  for (unsigned r = 0; r < (unsigned)kCS; ++r) st_remote_u32(map_remote(smem_addr(ticket), r), t);
}

// ---- solving block -------------------------------------------------------------------------------------
// early: the block has not waited for the kernel before this one yet, and its cluster has arrived at the cluster barrier
// that says that the shared memory of all its blocks is ready.  It draws its ticket here; anything but 0 sends it back.
template <class G, bool COLTYPE, bool AL>
__device__ __forceinline__ unsigned solve_block(const Args<typename G::T>& p, Block<typename G::T>& b, int rank, bool early, unsigned* ticket) {
  using T = typename G::T;
  using TL = Tile<G>;
  using P = typename TL::P;
  constexpr int NB = G::NB, V = G::V, WPE = Words<T>::N, SPB = NB / kStrip, NEAR = G::NEAR;
  const int W = p.W;
  constexpr int RS = TL::RS, CP = TL::CP, H = TL::H, NPK = TL::NPK;
  // Near tiles of column-type views are multiplied as they lie in memory: a lane holds V rows of op(A), a warp NB / 8 columns,
  // SG at a time, and the sums run across the warps.
  constexpr int LR = NB / V, SG = 32 / LR, JT = NB / (kCW * SG);
  static_assert(JT == NPK, "both tile layouts give a thread the same number of packs");
  // (The word itself is awaited, not the cluster barrier behind it: that takes 400 cycles even where everyone has arrived.)
  auto my_ticket = [&]() {
    __shared__ unsigned s_mine;
    if (b.tid == 0) {
      unsigned t = *(volatile unsigned*)ticket;
      while (t == kNoTicket && b.wt.again()) t = *(volatile unsigned*)ticket;
      s_mine = t == kNoTicket ? 0xffffffffu : t;
    }
    bar_block();
    return s_mine;
  };
  auto enter = [&]() {
    grid_dep_wait();
    grid_dep_launch();
  };
  auto draw = [&]() {
    __syncwarp();
    cluster_wait();
    if (rank == 0 && b.tid == 0) draw_ticket(p, ticket, true);
  };
  if (rank >= p.K) {
    if (early) {
      enter();
      draw();
      if (const unsigned t = my_ticket()) return t;
    }
    b.leave(p.ctl);
    return 0u;
  }
  const Scratchpad<G> pad(b.big + Smem<G>::NEAR_ELEMS);  // behind the near-tile ring
  const unsigned at = smem_off(pad.S);
  const int rg = b.tid >> 4, cg = b.tid & 15;
  const int row = TL::row(b.tid);
  const bool owner = cg % (16 / RS) == 0;
  const bool transposed = Diag<G, COLTYPE, AL>::transposed(p.backward);

  // near tiles: the sequence (k, w), k = rank, rank + kCS, ..., w = 2 .. min(W, K - 1 - k), NEAR tiles ahead
  int nk = rank, nw = 2, nslot = 0;
  // near tiles multiplied (so far); a slot is filled by a thread of its own (asker), which knows of its copies how many it has
  // begun and how many have landed.  (By one thread, four to six copies took 0.5 us; the first warps draw the ticket.)
  int used = 0, asked = 0, landed = 0;
  auto asker = [&](int slot) { return b.tid == kCT - 32 - slot * 32; };
  constexpr bool TMA = kTma && AL;
  auto near_width = [&](int k) { return min(W, p.K - 1 - k); };
  auto produce = [&]() {
    while (nk < p.K && nw > near_width(nk)) nk += kCS, nw = 2;
    if (TMA && nk < p.K) {
      const int I = mem_block(p, nk + nw), J = mem_block(p, nk);
      if (asker(nslot) && !*b.wt.dead) {
        mbar_arrive_expect(b.full + nslot, (unsigned)Smem<G>::NEAR_TILE);
        tma_load_2d(b.big + (size_t)nslot * NB * NB, b.map, (COLTYPE ? I : J) * NB, (COLTYPE ? J : I) * NB, b.full + nslot);
        ++asked;
      }
      ++nw;
    } else if (nk < p.K) {
      const int I = mem_block(p, nk + nw), J = mem_block(p, nk);
      const int li = block_len<NB>(p, I), lj = block_len<NB>(p, J);
      T* dst = b.big + (size_t)nslot * NB * NB + (size_t)b.tid * V;
      if (!AL && li == NB && lj == NB) {
        const int ru = COLTYPE ? b.warp * JT * SG : 2 * b.warp * RS;  // a warp's packs: SG stored rows, or (halves of) two
        const T* src = p.a + ((int64_t)(COLTYPE ? J : I) * NB + ru) * p.lda + (int64_t)(COLTYPE ? I : J) * NB + b.lane;
        dst -= b.lane * (V - 1);
        __syncwarp();
#pragma unroll
        for (int m = 0; m < NPK; ++m)
#pragma unroll
          for (int e = 0; e < V; ++e) {
            const int r = COLTYPE ? m * SG + e * 32 / NB : e * 32 / H * RS + m / CP, c = COLTYPE ? e * 32 % NB : (m % CP) * H + e * 32 % H;
            cp_async_elem<sizeof(T)>(dst + (size_t)m * kCT * V + e * 32, src + r * p.lda + c, true);
          }
      } else
#pragma unroll
      for (int m = 0; m < NPK; ++m) {
        const int r = COLTYPE ? (b.warp * JT + m) * SG + b.lane / LR : rg * RS + m / CP, c = COLTYPE ? b.lane % LR * V : (m % CP) * H + cg * V;
        const int rows = COLTYPE ? lj : li, cols = COLTYPE ? li : lj;
        const T* src = p.a + ((int64_t)(COLTYPE ? J : I) * NB + r) * p.lda + (int64_t)(COLTYPE ? I : J) * NB + c;
        if (AL && li == NB && lj == NB) cp_async16_full(dst + (size_t)m * kCT * V, src);
        else copy_pack<T, AL>(dst + (size_t)m * kCT * V, src, r < rows ? min(V, max(0, cols - c)) : 0, p.a);
      }
      ++nw;
    }
    if (!TMA) cp_async_commit();
    nslot = nslot + 1 == NEAR ? 0 : nslot + 1;
  };
  int rslot = 0;  // ring position of the tile that is multiplied next
  // The next near tile -> registers, in whole rows (columns, of column-type views) of the tile or as the threads copied it.
  auto near_tile = [&](P (&t)[NPK]) {
    const T* src = b.big + (size_t)rslot * NB * NB;
    if constexpr (TMA) {
      bool there = mbar_try_wait(b.full + rslot, (unsigned)(used / NEAR) & 1u);
      while (!there && b.wt.again()) there = mbar_try_wait(b.full + rslot, (unsigned)(used / NEAR) & 1u);
      if (asker(rslot) && there && !*b.wt.dead) ++landed;
      __syncwarp();
      if constexpr (!COLTYPE) {
        TL::from_rows(t, src, NB, b.tid);
      } else {
#pragma unroll
        for (int m = 0; m < NPK; ++m) t[m] = *reinterpret_cast<const P*>(src + (size_t)((b.warp * JT + m) * SG + b.lane / LR) * NB + b.lane % LR * V);
      }
    } else {
      cp_async_wait<NEAR - 1>();
      if (!AL) __syncwarp();
#pragma unroll
      for (int m = 0; m < NPK; ++m) t[m] = *reinterpret_cast<const P*>(src + ((size_t)m * kCT + b.tid) * V);
    }
    rslot = rslot + 1 == NEAR ? 0 : rslot + 1;
    ++used;
  };
  // No copy may arrive once the ring serves something else.  (All have landed where no wait ran out and no other cluster solves.)
  auto drain = [&]() {
    if constexpr (TMA) {
      static_assert(NEAR < kCW, "a warp for each slot");
      const int slot = kCW - 1 - b.warp;
      for (; landed < asked; ++landed)
        for (int spin = 0; spin < (1 << 16) && !mbar_try_wait(b.full + slot, (unsigned)landed & 1u); ++spin) {
        }
    }
  };

  // The chain is at the first rows before their tiles are premultiplied.  (A copy and two solves, us, from row 1 / 3 on: double n = 608 29.5 /
  // 28.4, 1024 37.5 / 36.9, 2048 59.2 / 58.2; float 1000 35.3 / 34.1, 1500 45.4 / 43.7.)
  const bool premultiplied = G::PM && p.pm > 0 && rank >= 3;
  P inv[NPK], nxt[NPK];  // inv(D_k), and beside it inv(D_k) A(k, k-1) -- or that tile, or A(k+1, k) where tiles are not premultiplied
  // The tile at positions (i, j) of the solve order -> nxt.
  auto load_tile = [&](int i, int j) {
    if constexpr (G::PM) {  // (where it is not premultiplied)
      if (premultiplied || i != rank) fetch_tile<G, COLTYPE, AL>(p, at, mem_block(p, i), mem_block(p, j), b.tid);
      if constexpr (COLTYPE) TL::from_columns(nxt, pad.n, Inv<G>::SP, b.tid, [](const T* q) { return *reinterpret_cast<const P*>(q); });
      else TL::from_rows(nxt, pad.n, Inv<G>::SP, b.tid);
    } else {
    const int I = mem_block(p, i), J = mem_block(p, j);
    const int li = block_len<NB>(p, I), lj = block_len<NB>(p, J);
    const T* src = p.a + (int64_t)(COLTYPE ? J : I) * NB * p.lda + (int64_t)(COLTYPE ? I : J) * NB;
    if (AL && li == NB && lj == NB) {
      if constexpr (!COLTYPE) {
#pragma unroll
        for (int m = 0; m < NPK; ++m) nxt[m] = ld_nc<T, V>(src + (rg * RS + m / CP) * p.lda + (m % CP) * H + cg * V);
      } else {  // packs run along op(A)'s rows: transposed on the way into the registers
        TL::from_columns(nxt, src, p.lda, b.tid, [](const T* q) { return ld_nc<T, V>(q); });
      }
    } else {
#pragma unroll
      for (int m = 0; m < NPK; ++m)
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const int r = rg * RS + m / CP, c = (m % CP) * H + cg * V + e;
          nxt[m].v[e] = r < li && c < lj ? __ldg(src + (COLTYPE ? c * p.lda + r : r * p.lda + c)) : T(0);
        }
    }
    }
  };
  // A(k+1, k) into L2, ahead of load_tile.
  auto prefetch_next = [&](int k) {
    if (k + 1 >= p.K) return;
    const int I = mem_block(p, k + 1), J = mem_block(p, k), R = COLTYPE ? J : I, Q = COLTYPE ? I : J;
    constexpr int LINES = NB * (int)sizeof(T) / 128;  // of a stored row of the tile
    const int rows = block_len<NB>(p, R), cols = block_len<NB>(p, Q);
#pragma unroll
    for (int i = 0; i < (NB * LINES + kCT - 1) / kCT; ++i) {
      const int r = (b.tid + i * kCT) / LINES, c = (b.tid + i * kCT) % LINES * (128 / (int)sizeof(T));
      if (r < rows && c < cols) prefetch_l2(p.a + ((int64_t)R * NB + r) * p.lda + (int64_t)Q * NB + c);
    }
  };

  const unsigned slots = smem_addr(b.slots);
  int par = 0;  // set of cross-warp sums
  T bk = T(0);  // this thread's element of the right-hand side
  // b_k less the sums of the rows before, those of rows k - W .. k - first by the cluster, the newest last -> rs
  // (All but the newest one are taken from b without rounding in between: a block row's right-hand side carries fewer rounding
  // errors than when each was rounded, and one addition stands in the chain.)
  auto gather_rhs = [&](int k, int first) {
    u64 wd[WPE];
    double hi = (double)bk, lo = 0.;
    auto take = [&](T v) {
      if constexpr (sizeof(T) == 4) {
        hi -= (double)v;
      } else {  // D. Knuth's sum with its error
        const double s = hi - v, b1 = hi - s;
        lo += (hi - (s + b1)) + (b1 - v);
        hi = s;
      }
    };
    auto sum_of = [&](int w) {
      const unsigned q = slots + (unsigned)(((w - 1) * NB + b.tid) * WPE * 8);
      ld_slot(q, wd);
      while (!tagged(wd, (unsigned)k + 1u)) {
        if (!b.wt.again()) break;
        ld_slot(q, wd);
      }
      return decode(wd, T(0));
    };
    if (k > W) {  // the streaming blocks' part
      const u64* q = p.far + ((int64_t)k * NB + b.tid) * WPE;
      ld_gpu(q, wd);
      while (!tagged(wd, p.tag)) {
        if (!b.wt.again()) break;
        ld_gpu(q, wd);
      }
      take(decode(wd, T(0)));
    }
#pragma unroll 1
    for (int w = min(W, k); w > first; --w) take(sum_of(w));
    const T r = (T)(isfinite(lo) ? hi + lo : hi);  // (with hi infinite the error is NaN)
    b.rs[b.tid] = k >= first ? r - sum_of(first) : r;
  };
  auto x_word = [&](int i) { return TL::x_word(slots, i); };
  // This thread's words of x_(k-1) as the neighbour stored them, and whether all are there.
  auto look_at_x = [&](u64 (&w)[CP][4], int k) {
    bool ok = true;
#pragma unroll
    for (int h = 0; h < CP; ++h) {
      const unsigned q = slots + (unsigned)((h * 32 + cg) * 16);
      ld_slot2(q, w[h][0], w[h][1]);
      ld_slot2(q + 256, w[h][2], w[h][3]);
    }
#pragma unroll
    for (int h = 0; h < CP; ++h)
#pragma unroll
      for (int i = 0; i < 4; ++i) ok = ok && (unsigned)(w[h][i] >> 32) == (unsigned)k + 1u;
    return ok;
  };
  // -x_(k-1) from them
  auto negated = [&](P (&x)[CP], const u64 (&w)[CP][4]) {
    constexpr unsigned MINUS = 0x80000000u, LOW = WPE == 1 ? MINUS : 0u;
#pragma unroll
    for (int h = 0; h < CP; ++h) {
      uint4 u = make_uint4((unsigned)w[h][0] ^ LOW, (unsigned)w[h][1] ^ MINUS, (unsigned)w[h][2] ^ LOW, (unsigned)w[h][3] ^ MINUS);
      x[h] = *reinterpret_cast<const P*>(&u);
    }
  };
  // One block row.
  // What lies between the arrival of u_1 (x_(k-1)) and the departure of the next block's runs twice, the first time
  // without its effects while the row still waits for its sums: code that has not run for microseconds is
  // fetched at a third of the speed at which it executes (u_1 to u_1 0.85 us -> 0.55 us in float).
  // have: nxt is premultiplied; later: near tiles to ask for once x_k is out; inverse: where inv came from, null: from S
  auto solve_row = [&](int k, bool have, int later, const T* inverse) {
    const int I = mem_block(p, k), li = block_len<NB>(p, I), wn = near_width(k);
    u64 wd[WPE];
    P cur[NPK], xv[CP];
    bool pub = false, fine = true;
    T xk;
    // The first near tile is waited for least of all: in registers ahead of the chain.
    const unsigned next = map_remote(G::PM ? x_word(row) : slots + (unsigned)(row * WPE * 8), (unsigned)((k + 1) % kCS));
    const bool ahead = G::PM && wn >= 2 && later == 0;
    if (ahead) near_tile(cur);
#pragma unroll 1
    for (int t = k < (G::PM ? 2 : 1) ? 1 : 0; t < 2; ++t) {  // (the first rows are waited for)
      const bool go = t == 1;
      if (go && b.tid < NB) gather_rhs(k, G::PM ? 2 : 1);
      if (go) bar_block();
      typename TL::Sums sums;
      TL::load_r(xv, b.rs, transposed, b.tid);
      if constexpr (G::PM) {
        // (x_(k-1) is often there before the sums of the rows further back)
        u64 w[CP][4];
        bool ok = look_at_x(w, k) || k == 0;
        const bool alive = !*b.wt.dead;
        TL::multiply(sums, inv, xv);
        while (go && !ok && b.wt.again()) {
#pragma unroll 1
          for (int i = 0; i < 4 && !ok; ++i) ok = look_at_x(w, k);  // (what again() does takes as long as a look)
        }
        pub = __all_sync(0xffffffffu, ok) && alive && go && k != p.debug_skip;
        negated(xv, w);
        if (go && !have) {  // nxt * x belongs on the other side of the inverse
          const T s = TL::product(nxt, xv, b.lane);
          bar_block();
          if (owner) b.rs[row] += s;
          bar_block();
          TL::load_r(xv, b.rs, transposed, b.tid);
          xk = TL::triangle(inv, xv, transposed, b.tid);
        } else {
          typename TL::Sums beside;
          TL::multiply(beside, nxt, xv);
          xk = TL::reduce(sums, beside, b.lane);
        }
        fine = !have || is_finite(xk);
        encode(xk, (unsigned)k + 2u, wd);
      } else {
        TL::multiply(sums, inv, xv);
        xk = TL::reduce(sums, b.lane);
        if (go) {
          if (owner) b.xs[row] = xk;
          bar_block();
        }
        TL::load_x(xv, b.xs, b.tid);
        const T u1 = TL::product(nxt, xv, b.lane);
        pub = go && !*b.wt.dead && k != p.debug_skip;
        encode(u1, (unsigned)k + 2u, wd);
      }
      // (what is not finite goes out after another look, below)
      st_slot_if(pub && owner && fine && k + 1 < p.K, next, wd);
      if (G::PM && go && owner) b.xs[row] = xk;
      encode(xk, p.tag, wd);
      st_gpu_if(pub && owner && fine, p.xbuf + ((int64_t)k * NB + row) * WPE, wd);
      st_val_if(pub && owner && fine && row < li, p.x + ((int64_t)I * NB + min(row, li - 1)) * p.incx, xk);
    }
    if constexpr (G::PM) {
      const bool again = pub && owner && !fine;
      __syncwarp();
      if (__builtin_expect(__syncthreads_or((int)again), 0))
        solve_apart<G, COLTYPE>(p, inverse, at, slots, smem_off(b.rs), smem_off(b.red + b.warp * NB), k, b.tid, transposed, again, xk);
    }
#pragma unroll 1
    for (int i = 0; i < later; ++i) produce();
#pragma unroll 1
    for (int w = 2; w <= wn; ++w) {
      if (w > 2 || !ahead) near_tile(cur);
      const unsigned dst = map_remote(slots + (unsigned)((w - 1) * NB * WPE * 8), (unsigned)((k + w) % kCS));
      if constexpr (!COLTYPE) {
        TL::load_x(xv, b.xs, b.tid);
        encode(TL::product(cur, xv, b.lane), (unsigned)(k + w) + 1u, wd);
        st_slot_if(pub && owner, dst + (unsigned)(row * WPE * 8), wd);
      } else {
        P s;
#pragma unroll
        for (int e = 0; e < V; ++e) s.v[e] = T(0);
#pragma unroll
        for (int m0 = 0; m0 < JT; m0 += V) {
          P xc;
          if constexpr (SG == 1) {
            xc = *reinterpret_cast<const P*>(b.xs + b.warp * JT + m0);
          } else {
#pragma unroll
            for (int m = 0; m < V; ++m) xc.v[m] = b.xs[(b.warp * JT + m0 + m) * SG + b.lane / LR];
          }
#pragma unroll
          for (int m = 0; m < V; ++m)
#pragma unroll
            for (int e = 0; e < V; ++e) s.v[e] = cur[m0 + m].v[e] * xc.v[m] + s.v[e];
        }
        if constexpr (SG > 1) {
#pragma unroll
          for (int e = 0; e < V; ++e) s.v[e] = cross_group_sum<LR>(s.v[e]);
        }
        T* red = b.red + (size_t)par * kCW * NB;
        par ^= 1;
        if (SG == 1 || b.lane < LR) *reinterpret_cast<P*>(red + b.warp * NB + b.lane * V) = s;
        bar_block();
        if (b.tid < NB) {
          T u = T(0);
#pragma unroll
          for (int v = 0; v < kCW; ++v) u += red[v * NB + b.tid];
          encode(u, (unsigned)(k + w) + 1u, wd);
          st_slot_if(pub, dst + (unsigned)(b.tid * WPE * 8), wd);
        }
      }
      if (TMA && !COLTYPE) bar_block();  // (every thread has read the slot; column-type views: above)
      produce();
    }
    if (!G::PM && k + kCS < p.K) prefetch_next(k + kCS);
  };

  auto load_rhs = [&](int k) {
    const int I = mem_block(p, k);
    bk = b.tid < block_len<NB>(p, I) ? p.x[((int64_t)I * NB + b.tid) * p.incx] : T(0);
  };

  // First row: its diagonal block and what is beside it, and the ticket in the meantime.  (Off 16-byte boundaries most near tiles
  // are asked for later: a thread is held while it asks for more than arrives, for 0.3 to 1 us a tile.)
  if (early) enter();
  load_rhs(rank);
  if constexpr (G::PM) {
    if (rank > 0) {
      const int I = mem_block(p, rank), J = mem_block(p, rank - 1);
      stage_tile<G, COLTYPE, AL>(p.a, p.lda, I, J, block_len<NB>(p, I), block_len<NB>(p, J), pad.n, b.tid);
    }
  }
  const int I0 = mem_block(p, rank);
  Diag<G, COLTYPE, AL>::stage(p.a, p.lda, p.n, I0, p.backward, pad.s, b.tid);
  if (!G::PM) prefetch_next(rank);
  if (early) draw();
  constexpr int EARLY = TMA ? NEAR : 2;
#pragma unroll 1
  for (int i = 0; i < EARLY; ++i) produce();
  cp_async_wait<TMA ? 0 : EARLY>();
  pad.arrived(premultiplied, b.tid);
  bar_block();
  if (invert_block<G>(at, smem_off(b.red), p.unit, block_len<NB>(p, I0), b.tid)) invert_again<G, COLTYPE, AL>(p, at, I0, b.tid);
  bool have = true;  // (row 0: nothing to multiply)
  if constexpr (G::PM) {
    if (rank > 0) have = premultiplied && !premultiply<G, COLTYPE>(at, smem_off(pad.N), transposed, block_len<NB>(p, I0), block_len<NB>(p, mem_block(p, rank - 1)), b.tid);
  }
  if (early) {
    if (const unsigned t = my_ticket()) {  // another cluster solves
      drain();
      bar_block();
      return t;
    }
  }
#pragma unroll 1
  for (int k = rank; k < p.K; k += kCS) {
    // Inverse of the diagonal block: the first row's is formed here, the others come from the streaming
    // blocks -- or are formed here after all, when the block that should deliver one has not started.
    __shared__ int s_self;
    bool formed = true;
    if (k != rank) {
      if (b.tid == 0) {
        int self = p.H == 0 ? 2 : 0;  // bit 1: formed here, bit 0: a premultiplied tile comes with it
        if (!self) {
          u64 f;
          while ((unsigned)((f = ld_flag(p.flags + k)) >> 32) != p.tag) {
            if (!has_started(p, p.H - 1 - (k - kCS) % p.H)) {
              self = 2;
              break;
            }
            if (!b.wt.again()) break;
          }
          if (!self) self = (int)(f & 1);
        }
        s_self = self;
      }
      bar_block();
      load_rhs(k);
      formed = s_self == 2, have = s_self == 1;
      if (formed) form_inverse<G, COLTYPE, AL>(p, at, smem_off(b.red), mem_block(p, k), b.tid);
    }
    if (!G::PM && k + 1 < p.K) load_tile(k + 1, k);
    const T* src = p.winv + (int64_t)(k - kCS) * NB * NB * (G::PM && p.pm > 1 ? 2 : 1);
    if (formed) TL::inverse(inv, pad.S, transposed, b.tid);
    else TL::load(inv, src, b.tid);
    if constexpr (G::PM) {
      if (k == 0) {
#pragma unroll
        for (int m = 0; m < NPK; ++m) nxt[m] = P{};
      } else if (!have) {
        load_tile(k, k - 1);
      } else if (k == rank) {
        TL::from_rows(nxt, pad.N, Inv<G>::SP, b.tid);
      } else {
        TL::load(nxt, src + NB * NB, b.tid);
      }
    }
    // The first row's other near tiles: as many as there is time for before the chain arrives, the rest behind x.
    const int rest = k != rank ? 0 : NEAR - EARLY, now = min(rest, rank * 12 * 1024 / (int)Smem<G>::NEAR_TILE);
#pragma unroll 1
    for (int i = 0; i < now; ++i) produce();
    // Sums that no running block will deliver (cold path; asked late, so that blocks that start a little
    // after this one are not taken for missing).
    if (k > W && b.warp < SPB && (p.H == 0 || !has_started(p, ((k - W - 1) * SPB + b.warp) % p.H))) {
      const T s = slow_strip<G, COLTYPE>(p, k, b.warp, k - W, b.wt, b.lane);
      u64 wd[WPE];
      encode(s, p.tag, wd);
      st_gpu_if(!*b.wt.dead, p.far + ((int64_t)k * NB + b.warp * kStrip + b.lane) * WPE, wd);
    }
    if (k + kCS >= p.K) b.leave(p.ctl);
    solve_row(k, have, rest - now, formed ? nullptr : src);
  }
  cp_async_wait<0>();
  drain();
  return 0u;
}

// ---- kernel --------------------------------------------------------------------------------------------
// __grid_constant__: a function that is not inlined gets the arguments by reference, and without it every thread keeps a copy
// of them in local memory and reads that in the chain (n = 9008 in double 346 us a pair of solves, so 261).
template <class G, bool COLTYPE, bool AL>
__global__ void __launch_bounds__(kCT, 1) trsv_cluster_kernel(const __grid_constant__ Args<typename G::T> p, const __grid_constant__ CUtensorMap map) {
  using T = typename G::T;
  using SM = Smem<G>;
  constexpr int NB = G::NB, WPE = Words<T>::N;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ unsigned s_ticket;
  __shared__ int s_dead;
  __shared__ __align__(8) u64 s_full[G::NEAR];
  Block<T> b;
  b.big = reinterpret_cast<T*>(smem_raw);
  b.red = reinterpret_cast<T*>(smem_raw + SM::BIG);
  b.slots = reinterpret_cast<u64*>(smem_raw + SM::BIG + SM::REDTM);
  b.rs = reinterpret_cast<T*>(smem_raw + SM::BIG + SM::REDTM + SM::SLOTS);
  b.xs = b.rs + NB;
  b.left = b.aborted = ~0u;
  b.tid = (int)threadIdx.x, b.warp = b.tid >> 5, b.lane = b.tid & 31;
  b.wt.budget = p.wait_limit ? p.wait_limit : (1ull << 22);
  b.wt.abort_word = p.ctl + kCtlTrsvAbort;
  b.wt.device_status = p.device_status;
  b.wt.dead = &s_dead;
  const int rank = (int)cluster_rank();
  for (int i = b.tid; i < G::W * NB * WPE; i += kCT) b.slots[i] = 0ull;  // no stale word may look like one of this call
  if (b.tid < 2 * NB) b.rs[b.tid] = T(0);
  b.full = s_full;
  b.map = &map;
  if (kTma && AL && b.tid == kCT - 32) asm volatile("prefetch.tensormap [%0];" ::"l"(&map) : "memory");
  if (b.tid == 0) {
    s_dead = 0;
    s_ticket = kNoTicket;
    if (kTma && AL) {
      for (int s = 0; s < G::NEAR; ++s) mbar_init(&s_full[s], 1u);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
  }
  __syncwarp();
  cluster_arrive();  // (shared memory of the cluster is ready)
  const bool early = blockIdx.x < (unsigned)kCS;  // (the first cluster usually draws the first ticket)
  unsigned t = 0u;
  if (!early) {
    grid_dep_wait();
    grid_dep_launch();
    __syncwarp();
    cluster_wait();
    if (rank == 0 && b.tid == 0) draw_ticket(p, &s_ticket, false);
    cluster_sync_all();
    t = s_ticket;
  }
  if (t == 0u) t = solve_block<G, COLTYPE, AL>(p, b, rank, early, &s_ticket);
  if (t != 0u) {
    cp_async_wait<0>();
    if (t != 0xffffffffu) {
      b.leave(p.ctl);
      stream_block<G, COLTYPE, AL>(p, b, (int)(t - 1u) * kCS + rank);
    }
  }
  cluster_sync_all();  // no block leaves while a peer may still write into its shared memory
  // the last block to leave puts the counters back (not after an abort: the caller resets)
  if (b.tid == 0 && b.left == gridDim.x - 1 && b.aborted == 0u) {
    p.ctl[kCtlTrsvTicket] = 0u;
    p.ctl[kCtlTrsvDone] = 0u;
  }
}

// ---- host ----------------------------------------------------------------------------------------------
// Clusters of kCS blocks of this kernel that the device holds at once (cached per device; 0: none).
template <class G, bool COLTYPE, bool AL>
static int max_clusters() {
  static int cached[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (cached[dev] == 0) {
    auto kern = trsv_cluster_kernel<G, COLTYPE, AL>;
    int n = 0;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kCS;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(kCS);
    cfg.blockDim = dim3(kCT);
    cfg.dynamicSmemBytes = Smem<G>::TOTAL;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Smem<G>::TOTAL) != cudaSuccess ||
        cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess)
      n = 0;
    (void)cudaGetLastError();
    cached[dev] = n > 0 ? n : -1;
  }
  return cached[dev] > 0 ? cached[dev] : 0;
}

template <class G, bool COLTYPE, bool AL>
static int launch_cluster(const Launch& l, Args<typename G::T>& p, size_t tagged_bytes, bool* handled) {
  constexpr int SPB = G::NB / kStrip;
  int room = max_clusters<G, COLTYPE, AL>() - 1;
  if (room < 0) return B2_STATUS_OK;
  const int64_t cap = knob(kKnobTrsvStreams);
  if (cap >= 0 && cap < room) room = (int)cap;
  p.W = AL ? G::W : p.K <= G::KU ? G::WU : G::WL;
  // streaming blocks: no more than there are strips or diagonal blocks for
  const int strips = std::max(0, p.K - p.W - 1) * SPB, want = std::max(strips, p.K - kCS);
  const int streams = std::min(room, want <= 0 ? 0 : (want + kCS - 1) / kCS);
  p.H = streams * kCS;
  if (strips > kStrips * p.H && cap != 0) return B2_STATUS_OK;  // (no streaming blocks at all: a test's choice)
  CUtensorMap map = {};
  if (kTma && AL && !encode_tile_map(&map, p.a, p.lda, p.n, G::NB, G::NB)) return launch_cluster<G, COLTYPE, false>(l, p, tagged_bytes, handled);
  *handled = true;
  if (int st = trsv_forget_if_captured(l, tagged_bytes)) return st;
  launch_clusters(trsv_cluster_kernel<G, COLTYPE, AL>, (unsigned)((1 + streams) * kCS), (unsigned)kCS, dim3(kCT), Smem<G>::TOTAL, l.stream, p, map);
  return check_launch();
}

// Workspace of a solve of K block rows: published x and far sums, flags of the inverses -- what carries tags -- and the
// inverses, with the premultiplied tiles where there is room for them.
template <class G>
struct Scratch {
  size_t words, tagged, inverses, total;
  explicit Scratch(int64_t K) {
    constexpr size_t NB = G::NB;
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    words = up((size_t)K * NB * Words<typename G::T>::N * 8);
    tagged = 2 * words + up((size_t)K * 8);
    inverses = tagged + (size_t)std::max<int64_t>(0, K - kCS) * NB * NB * sizeof(typename G::T);
    total = G::PM ? 2 * inverses - tagged : inverses;
  }
};

// Last block rows whose tiles beyond the first turn are premultiplied off 16-byte boundaries.  There the streaming blocks, which have
// that to do first, are the slower ones while many strips need each tile; the chain waits for them and has time for two products.
// (Double, mean of four views, us a solve, all / none / the last 40 / 56 / 72 premultiplied: n = 7001 134.7 / 139.5 / 135.1 / 134.1 / 134.2, 8001 161.8 /
// 166.7 / 159.3 / 158.7 / 161.4, 10001 222.9 / 225.3 / 219.9 / 219.4 / 220.2, 11519 287.3 / 287.9 / 284.5 / 283.2 / 283.6.  The first 72 rows of 110 premultiplied
// instead of the last: 138.6.)
constexpr int kPremultiplyLast = 56;

// Block rows from which tiles are premultiplied: with fewer the chain is shorter than what that takes.  (A copy and both solves, us,
// without / with it: float n = 100 17.1 / 20.0, 200 20.8 / 22.3, 380 24.3 / 24.3, 450 31.0 / 29.1, 600 31.4 / 28.5; double 100 16.9 / 18.3, 250
// 21.3 / 21.5, 300 22.5 / 22.5, 380 24.5 / 23.7, 600 31.9 / 28.9.  And few rows' products are more exact as they were: the error
// in double at n = 100 and 300 is 5 and 3 % larger with it, from 700 on 5 to 8 % smaller than before them.)
template <typename T>
constexpr int64_t kPremultiplyFrom = sizeof(T) == 4 ? 7 : 6;

template <class G>
static int run_cluster(const Launch& l, bool coltype, Args<typename G::T>& p, bool* handled) {
  constexpr int NB = G::NB;
  const int64_t K = (p.n + NB - 1) / NB;
  if (K > (1 << 20)) return B2_STATUS_OK;
  const Scratch<G> w(K);
  if (w.inverses > l.scratch_bytes) return B2_STATUS_OK;
  const bool al = aligned_to(p.a, 16) && p.lda % G::V == 0;
  p.pm = K < kPremultiplyFrom<typename G::T> ? 0 : w.total <= l.scratch_bytes ? 2 : 1;
  p.pm_from = al ? 0 : (int)K - kPremultiplyLast;
  p.xbuf = reinterpret_cast<u64*>(l.scratch);
  p.far = reinterpret_cast<u64*>(l.scratch + w.words);
  p.flags = reinterpret_cast<u64*>(l.scratch + 2 * w.words);
  p.winv = reinterpret_cast<typename G::T*>(l.scratch + w.tagged);
  p.K = (int)K;
  if (coltype) return al ? launch_cluster<G, true, true>(l, p, w.tagged, handled) : launch_cluster<G, true, false>(l, p, w.tagged, handled);
  return al ? launch_cluster<G, false, true>(l, p, w.tagged, handled) : launch_cluster<G, false, false>(l, p, w.tagged, handled);
}

// Unknowns up to which float takes the short block rows: the start costs half as much (an inverse 3300 cycles instead of
// 10600) and a row 0.5 us instead of 0.8, but there are twice as many.  A copy and both solves, us, rows of 128 / 64 (row-major; column-major):
// n = 1024 37.4 / 35.6; 39.6 / 36.6, 1536 44.0 / 45.1; 46.3 / 46.0, 2048 51.5 / 54.1; 54.0 / 54.8, 2560 58.2 / 62.6; 60.4 / 63.4; off 16-byte boundaries, where the longer
// rows' tiles take long to copy, 1001 47.2 / 38.3; 49.2 / 38.8, 4001 95.3 / 88.6; 98.7 / 89.4, 4601 105.5 / 103.5; 110.5 / 105.1, 4801 (72 rows of 64 have two strips
// for some streaming blocks) 110.4 / 118.7; 114.7 / 118.9, 5301 122.8 / 129.1; 127.9 / 132.2.  (The error against a solve in double is 4 to 9 % smaller in rows of 128.)
constexpr int64_t kShortRows = 1536, kShortRowsUnaligned = 4608;

}  // namespace tc

size_t trsv_cluster_scratch(int64_t n, size_t elem_bytes) {
  using namespace tc;
  auto rows = [&](int64_t m, int64_t nb) { return (m + nb - 1) / nb; };
  if (elem_bytes == 4) return std::max(Scratch<F128>(rows(n, 128)).total, Scratch<F64>(rows(std::min(n, kShortRowsUnaligned), 64)).total);
  return Scratch<D64>(rows(n, 64)).total;
}

template <typename T>
int trsv_cluster_try(const Launch& l, bool coltype, bool backward, bool unit, int64_t n, const T* a, int64_t lda, T* xbase, int64_t incx,
                     unsigned tag, bool* handled) {
  using namespace tc;
  *handled = false;
  Args<T> p = {};
  p.a = a;
  p.lda = lda;
  p.n = n;
  p.x = xbase;
  p.incx = incx;
  p.ctl = l.ctl;
  p.backward = backward;
  p.unit = unit;
  p.tag = tag;
  p.wait_limit = l.wait_limit;
  p.device_status = l.device_status;
  p.debug_skip = (int)knob(kKnobTrsvDebugSkip);
  p.debug_late = (int)knob(kKnobTrsvDebugLate);
#ifdef B2_DEBUG_BOUNDS
  {  // (this translation unit has its own copy of the range table)
    Launch lc = l;
    B2_DBG_COMMIT(lc);
  }
#endif
  if constexpr (sizeof(T) == 8) {
    return run_cluster<D64>(l, coltype, p, handled);
  } else {
    const bool al = aligned_to(a, 16) && lda % 4 == 0;
    const int64_t k = knob(kKnobTrsvShortRows), most = k >= 0 ? k : al ? kShortRows : kShortRowsUnaligned;
    if (n <= most) {  // (rows of 128 need no inverses where rows of 64 need too many for the workspace)
      const int st = run_cluster<F64>(l, coltype, p, handled);
      if (st != B2_STATUS_OK || *handled) return st;
    }
    return run_cluster<F128>(l, coltype, p, handled);
  }
}

template int trsv_cluster_try<float>(const Launch&, bool, bool, bool, int64_t, const float*, int64_t, float*, int64_t, unsigned, bool*);
template int trsv_cluster_try<double>(const Launch&, bool, bool, bool, int64_t, const double*, int64_t, double*, int64_t, unsigned, bool*);

}  // namespace b2
