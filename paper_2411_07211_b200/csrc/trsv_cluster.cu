// trsv, cluster kernel: solve op(A) x = b in place (Section 6.2.2; same option space as trmv).
//
// The unknowns are cut into block rows of NB (128 float / 64 double), numbered in solve order.  The
// chain x_0 -> x_1 -> ... is the only sequential part; what it costs is the hand-over from one block
// row to the next, about 1 us through L2 and 0.2 us through the shared memory of a cluster.  So ONE
// cluster of kCS blocks walks the whole chain, and the other blocks of the grid stream the matrix:
//
//   solving block (rank c of the first cluster; block rows k = c, c + kCS, ...)
//     r   = b_k - far_k - u_W - ... - u_1      far_k from the streaming blocks, u_w = A(k, k-w) x(k-w)
//                                              from the cluster blocks that solved the rows before
//     x_k = inv(D_k) r                         inverse in registers
//     u   = A(k+w, k) x_k, w = 1 .. W          stored straight into the shared memory of the block that
//                                              owns row k + w (A(k+1, k) from registers, the others
//                                              through a shared-memory ring of asynchronous copies)
//     Between u_1's arrival in row k and its arrival in row k + 1 lie two register products, two
//     block barriers and one store into a neighbour's shared memory.
//   streaming block: 32-row strips of op(A), dealt out cyclically; at each step it multiplies the tiles
//     (strip, j), (strip, j + 1) of each of its strips that still needs them by x_j and x_(j+1) and keeps
//     the sums in registers.  Tile data does not depend on the solve, so a ring of 192 KB is always in
//     flight: every thread copies exactly the packs it later reads, so the ring needs no barrier.  A strip
//     of row k is complete after x(k-W-1); its sums are published W steps before the chain needs them,
//     which hides the two trips through L2.
//   The streaming blocks first invert the diagonal blocks of the rows beyond the first kCS.
// The blocks of the first cluster start as solving ones -- they request and invert their diagonal blocks -- before they know
// their ticket; the others draw theirs a little later, and if the first cluster is late, one of them solves.
//
// Values cross blocks as tagged words (payload and ready flag in one store; the tag is unique per call
// in global memory, the row number in shared memory); consumers poll the data itself.  Every wait is
// bounded.  No co-residency is assumed: roles go by tickets drawn when a cluster starts, a streaming
// block only waits for the solving cluster (which drew the first ticket), and the solving cluster does
// the work of a streaming cluster that has not started yet itself, in the same order of additions.
//
// What bounds it: the chain, 0.94 us per block row in float (two products 0.55 us, the store into the neighbour and its
// poll 0.2 us, waiting for sums the rest) and 0.75 us in double, after 6 us (double) to 14 us (float, large n) until the first
// row is solved: its diagonal block is there after 2 to 3 us, asked for ahead of the near tiles and of the cluster's role, and
// inverted in 1.5 / 5.4 us (trsv_cluster.cuh; 14 us until the inverse was there before both).  From n = 11520 on in
// double the streaming blocks (112 of them, the clusters leave 20 SMs idle), 5 TB/s.  A copy and both solves, us, before the
// early start, the inverse by matrix instructions and what NearRows and stream_block say / now: float n = 80 33.5 / 24.8,
// 1000 52.1 / 44.7, 11520 224 / 208, 3001 92.6 / 82, 8191 236 / 230; double 80 27.3 / 18.1, 1024 50.5 / 42.8, 9008 275 / 262, 8191 336 / 329.
// Against the sub-block kernel of trsv_front.cu, per solve, N / T views, before that: float n = 1024 22.5 / 25.6 us (27 / 27), 11520
// 104 / 116 us (141 / 134); double n = 1024 24.4 / 24.9 us (32 / 30), 11520 164 / 160 us (238 / 228); rows off 16-byte
// boundaries, against the block-row kernel: float n = 4097 61 / 63 us (103 / 128), double n = 4097 65 / 67 us (126 / 116).
// Tried: clusters of 8 (column-type views 40 % slower in float: a block's pass over its near tiles takes
// longer than its turn), the near tiles on the receiving side (0.8 us more per row: the last of them then
// stands in the chain), one tile per ring slot (streaming alone 84 us instead of 51 us at n = 11520).
#include <algorithm>

#include "trsv_cluster.cuh"
#include "trsv_front.cuh"

namespace b2 {
namespace tc {

constexpr int kCS = 16;         // blocks per cluster (the opt-in size: 16 turns hide a row's preparation)
constexpr int kStrip = 32;      // rows of op(A) in a strip
constexpr int kDepth = 6;       // slots of a streaming block's ring, two tiles (32 KB) each
constexpr int kStrips = 12;     // strips per streaming block at most
constexpr int kTilePacks = 4;   // packs of a strip's tile per thread
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
  T* winv;           // [K - kCS][NB * NB] inverses of the diagonal blocks beyond the first kCS (of their transposes: Diag)
  unsigned* flags;   // [K] call tag once winv[k] is complete
  unsigned* ctl;
  int K;             // block rows
  int H;             // streaming blocks of the grid
  int backward, unit;
  unsigned tag;
  u64 wait_limit;
  int* device_status;
  int debug_skip;
  int debug_late;  // test hook: polls for which the first cluster lets another one draw the first ticket
};

// Shared memory: one region that is the solving block's near-tile ring and inversion scratch or the
// streaming block's tile ring, then the small arrays.
template <typename T>
struct Smem {
  static constexpr int NB = Geo<T>::NB, WPE = Words<T>::N;
  static constexpr size_t NEAR_TILE = (size_t)NB * NB * sizeof(T);
  static constexpr size_t NEAR_ELEMS = (size_t)Geo<T>::NEAR * NB * NB;
  static constexpr size_t SOLVE = Geo<T>::NEAR * NEAR_TILE + sizeof(T) * Inv<T>::S_ELEMS;
  static constexpr size_t SLOT = 2 * (size_t)kTilePacks * kCT * 16;
  static constexpr size_t STREAM = kDepth * SLOT;
  static constexpr size_t BIG = SOLVE > STREAM ? SOLVE : STREAM;
  static constexpr size_t RED = 2 * (size_t)kCW * NB * sizeof(T);  // cross-warp sums, two sets (also the inversion's Tm)
  static constexpr size_t TM = sizeof(T) * Inv<T>::TM_ELEMS;
  static constexpr size_t REDTM = RED > TM ? RED : TM;
  static constexpr size_t SLOTS = (size_t)Geo<T>::W * NB * WPE * 8;
  static constexpr size_t VECS = 4 * NB * sizeof(T);  // r, x of a row; two pairs of x blocks
  static constexpr size_t TOTAL = BIG + REDTM + SLOTS + VECS;
  // a streaming block inverts in the last slots of its ring, while the first ones fill
  static constexpr int FREE_SLOTS = (int)((STREAM - sizeof(T) * Inv<T>::S_ELEMS) / SLOT);
};

template <typename T>
struct Block {  // what both roles share
  T *big, *red, *rs, *xs;
  u64* slots;
  Waiter wt;
  int tid, warp, lane;
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
template <typename T>
__device__ __forceinline__ int block_len(const Args<T>& p, int I) { return (int)min((int64_t)Geo<T>::NB, p.n - (int64_t)I * Geo<T>::NB); }

// Whether the cluster that holds streaming block h has started (its ticket has been drawn).
template <typename T>
__device__ __forceinline__ bool has_started(const Args<T>& p, int h) {
  return ld_flag(p.ctl + kCtlTrsvTicket) > (unsigned)(1 + h / kCS);
}

// ---- a strip's tile ------------------------------------------------------------------------------------
// Sums of a thread.  Row-type views (op(A)'s rows contiguous): warp w holds rows 4w .. 4w + 3 of the
// strip, a lane V columns of each, one sum per row.  Column-type views: the warp's lanes run along the
// strip (contiguous in memory), over NB / 8 columns of the tile; V sums per lane, one per row of op(A).
template <typename T, bool COLTYPE>
struct Strip {
  static constexpr int NB = Geo<T>::NB, V = Geo<T>::V;
  static constexpr int NA = COLTYPE ? V : kTilePacks;
  static constexpr int LPR = kStrip / V, GR = 32 / LPR;  // column-type: lanes along the strip, stored rows per instruction
  static_assert(kCW * kTilePacks * GR == NB, "column-type: every stored row of the tile exactly once");

  // address and number of existing elements of pack q of this thread
  __device__ __forceinline__ static const T* pack_ptr(const Args<T>& p, int I, int sub, int J, int warp, int lane, int q, int* valid) {
    int64_t r, c;
    int rl, cl;
    if (!COLTYPE) {
      const int i = sub * kStrip + warp * kTilePacks + q;
      r = (int64_t)I * NB + i, c = (int64_t)J * NB + lane * V;
      rl = block_len(p, I) - i, cl = block_len(p, J) - lane * V;
    } else {
      const int j = warp * (NB / kCW) + lane / LPR + GR * q, i = sub * kStrip + (lane % LPR) * V;
      r = (int64_t)J * NB + j, c = (int64_t)I * NB + i;
      rl = block_len(p, J) - j, cl = block_len(p, I) - i;
    }
    *valid = rl > 0 ? (cl < 0 ? 0 : cl > V ? V : cl) : 0;
    return p.a + r * p.lda + c;
  }
  // this thread's values of x for every tile of a block column
  static constexpr int NX = COLTYPE ? kTilePacks : V;
  __device__ __forceinline__ static void load_x(T (&x)[NX], const T* xv, int warp, int lane) {
    if constexpr (!COLTYPE) {
      ld_pack(xv + lane * V, x);
    } else {
#pragma unroll
      for (int q = 0; q < kTilePacks; ++q) x[q] = xv[warp * (NB / kCW) + lane / LPR + GR * q];
    }
  }
  __device__ __forceinline__ static void add(T (&acc)[NA], const Pack<T, V> (&m)[kTilePacks], const T (&x)[NX]) {
#pragma unroll
    for (int q = 0; q < kTilePacks; ++q)
#pragma unroll
      for (int e = 0; e < V; ++e) {
        if (!COLTYPE) acc[q] = m[q].v[e] * x[e] + acc[q];
        else acc[e] = m[q].v[e] * x[q] + acc[e];
      }
  }
};

// Complete row sums of a strip from its threads' sums -> far words of block row k.  All threads.
template <typename T, bool COLTYPE>
__device__ __forceinline__ T strip_rows(const T (&sum)[Strip<T, COLTYPE>::NA], T* red, int warp, int lane, int* row) {
  using ST = Strip<T, COLTYPE>;
  if constexpr (!COLTYPE) {  // every eighth lane gets a row
    T v[kTilePacks];
#pragma unroll
    for (int q = 0; q < kTilePacks; ++q) v[q] = sum[q];
    const T s = multi_group_sum<32, kTilePacks>(v, lane);
    constexpr int LPV = 32 / kTilePacks;
    *row = lane % LPV == 0 ? warp * kTilePacks + lane / LPV : -1;
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

// acc[s] += tiles * x with s known at run time (the sums stay in registers); both: the second tile counts;
// done: the sums, when `last`.
template <typename T, bool COLTYPE, int I>
__device__ __forceinline__ void add_to(T (&acc)[kStrips][Strip<T, COLTYPE>::NA], int s, const Pack<T, Geo<T>::V> (&m)[2][kTilePacks],
                                       const T (&x)[2][Strip<T, COLTYPE>::NX], bool both, bool last, T (&done)[Strip<T, COLTYPE>::NA]) {
  if (s == I) {
    Strip<T, COLTYPE>::add(acc[I], m[0], x[0]);
    if (both) Strip<T, COLTYPE>::add(acc[I], m[1], x[1]);
    if (last) {
#pragma unroll
      for (int e = 0; e < Strip<T, COLTYPE>::NA; ++e) done[e] = acc[I][e];
    }
  } else if constexpr (I + 1 < kStrips) {
    add_to<T, COLTYPE, I + 1>(acc, s, m, x, both, last, done);
  }
}

// Diagonal block I once more, from the matrix (cold path; all copies of this thread that are in flight are waited for).
template <typename T, bool COLTYPE, bool AL>
__device__ __noinline__ void invert_again(const Args<T>& p, unsigned s_off, int I, int tid) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* const S = reinterpret_cast<T*>(smem_raw + s_off);
  Diag<T, COLTYPE, AL>::stage(p.a, p.lda, p.n, I, p.backward, S, tid);
  cp_async_wait<0>();
  bar_block();
  invert_rows<T>(S, p.unit, block_len(p, I), tid);
}

// ---- streaming block -----------------------------------------------------------------------------------
template <typename T, bool COLTYPE, bool AL>
__device__ __forceinline__ void stream_block(const Args<T>& p, Block<T>& b, int h) {
  using ST = Strip<T, COLTYPE>;
  constexpr int NB = Geo<T>::NB, V = Geo<T>::V, WPE = Words<T>::N, SPB = NB / kStrip;  // strips per block row
  constexpr int W = NearRows<T, AL>::W;
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
  const T* const at = p.a + (COLTYPE ? (int64_t)(b.warp * (NB / kCW) + b.lane / ST::LPR) * p.lda + (b.lane % ST::LPR) * V
                                     : (int64_t)(b.warp * kTilePacks) * p.lda + b.lane * V);
  const T* const uat = p.a + (COLTYPE ? (int64_t)(b.warp * (NB / kCW)) * p.lda : (int64_t)(b.warp * kTilePacks) * p.lda) + b.lane;
  const int64_t step_a = COLTYPE ? ST::GR * p.lda : p.lda, step_e = COLTYPE ? p.lda : 32;  // (step_e: see copy_warp)
  const int64_t jstep = (COLTYPE ? p.lda : 1) * (p.backward ? -NB : NB);  // from a block column to the next in solve order
  const int64_t j0off = (COLTYPE ? p.lda : 1) * (int64_t)mem_block(p, 0) * NB;
  auto produce = [&]() {
    if (pj <= jmax) {
      T* dst = b.big + ((size_t)(pslot * 2 * kTilePacks) * kCT + b.tid) * V;
      const bool both = pj < s_last[ps];
      const bool whole = ragged < 0 || (p.backward ? pj > 0 : (q0 + ps * H) / SPB != ragged);
      if (whole) {
        const int64_t tile = s_base[ps] + j0off + pj * jstep;
        if constexpr (AL) {
          const T* src = at + tile;
#pragma unroll
          for (int r = 0; r < kTilePacks; ++r) cp_async16_full(dst + (size_t)r * kCT * V, src + r * step_a);
          if (both) {
#pragma unroll
            for (int r = 0; r < kTilePacks; ++r) cp_async16_full(dst + (size_t)(kTilePacks + r) * kCT * V, src + jstep + r * step_a);
          }
        } else {
          const T* src = uat + tile;
          dst -= b.lane * (V - 1);
#pragma unroll
          for (int r = 0; r < kTilePacks; ++r) copy_warp(dst + (size_t)r * kCT * V, src + r * step_a, step_e);
          if (both) {
#pragma unroll
            for (int r = 0; r < kTilePacks; ++r) copy_warp(dst + (size_t)(kTilePacks + r) * kCT * V, src + jstep + r * step_a, step_e);
          }
        }
      } else {
        const int q = q0 + ps * H;
#pragma unroll 1
        for (int r = 0; r < (both ? 2 : 1) * kTilePacks; ++r) {
          int valid;
          const T* src = ST::pack_ptr(p, mem_block(p, q / SPB), q % SPB, mem_block(p, pj + r / kTilePacks), b.warp, b.lane, r % kTilePacks, &valid);
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
    T* M = reinterpret_cast<T*>(reinterpret_cast<unsigned char*>(b.big) + Smem<T>::STREAM) - Inv<T>::S_ELEMS;
    const int I = mem_block(p, k);
    Diag<T, COLTYPE, AL>::stage(p.a, p.lda, p.n, I, p.backward, M, b.tid);
    if (filled == 0) {
#pragma unroll 1
      for (; filled < Smem<T>::FREE_SLOTS; ++filled) produce();
      cp_async_wait<Smem<T>::FREE_SLOTS>();
    } else {
      cp_async_wait<0>();
    }
    bar_block();
    if (invert_block<T>(smem_off(M), smem_off(b.red), p.unit, block_len(p, I), b.tid)) invert_again<T, COLTYPE, AL>(p, smem_off(M), I, b.tid);
    T* dst = p.winv + (int64_t)(k - kCS) * NB * NB;
#pragma unroll 2
    for (int idx = b.tid; idx < NB * NB / V; idx += kCT) {
      T v[V];
      ld_pack(M + (idx / (NB / V)) * Inv<T>::SP + (idx % (NB / V)) * V, v);
      st_pack(dst + idx * V, v);
    }
    __threadfence();
    bar_block();
    if (b.tid == 0) st_flag(p.flags + k, p.tag);
  }
#pragma unroll 1
  for (; filled < kDepth - 1; ++filled) produce();

  // x_j and x_(j+1): one word per thread (a block's x is 128 words in both precisions), loaded a step ahead; into
  // one of two shared-memory buffers, then one block barrier per step.  (x_(j+1) is there long before the
  // row that a strip with last tile j belongs to is due.)
  static_assert(2 * NB * WPE == kCT, "one word per thread");
  const u64* xsrc = p.xbuf + b.tid;
  u64 xw[1];
  if (jmax >= 0) ld_gpu(xsrc, xw);
  int slot = 0, lo = 0, par = 0;
  auto finish = [&](int q, const T (&sum)[ST::NA]) {  // strip q is complete
    int row;
    const T v = strip_rows<T, COLTYPE>(sum, b.red + par * (kCW * kStrip), b.warp, b.lane, &row);
    par ^= 1;
    u64 wd[WPE];
    encode(v, p.tag, wd);
    st_gpu_if(row >= 0 && !*b.wt.dead, p.far + ((int64_t)(q / SPB) * NB + (q % SPB) * kStrip + max(row, 0)) * WPE, wd);
  };
#pragma unroll 1
  for (int j = 0; j <= jmax; j += 2) {
    T* xv = b.rs + (j & 2) * NB;  // (xs: four blocks)
    auto receive = [&]() {
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
    const bool alone = sizeof(T) == 4 && AL && s_last[lo] == j;
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
      const T* src = b.big + ((size_t)(slot * 2 * kTilePacks) * kCT + b.tid) * V;
      slot = slot + 1 == kDepth ? 0 : slot + 1;
      cp_async_wait<kDepth - 1>();
      if (!AL) __syncwarp();
      Pack<T, V> m[2][kTilePacks];
#pragma unroll
      for (int r = 0; r < 2 * kTilePacks; ++r)
        m[r / kTilePacks][r % kTilePacks] = *reinterpret_cast<const Pack<T, V>*>(src + (size_t)r * kCT * V);
      T done[ST::NA];
      add_to<T, COLTYPE, 0>(acc, s, m, x, j < last_j, last_j - j <= 1, done);
      if (last_j - j <= 1) finish(q0 + s * H, done);
    }
  }
  cp_async_wait<0>();
}

// Row sums of a strip that no running block will deliver, by one warp of the solving block (lane i:
// row i of the strip), with the additions of a streaming block in the same order.
template <typename T, bool COLTYPE>
__device__ __noinline__ T slow_strip(const Args<T>& p, int k, int sub, int jend, Waiter wt, int lane) {
  using ST = Strip<T, COLTYPE>;
  constexpr int NB = Geo<T>::NB, V = Geo<T>::V, WPE = Words<T>::N;
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
      for (int r = 0; r < kTilePacks; ++r) {
        int valid;
        const T* src = ST::pack_ptr(p, I, sub, J, w, lane, r, &valid);
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const T m = e < valid ? __ldg(src + e) : T(0);
          if (!COLTYPE) acc[r] = m * x_at(lane * V + e) + acc[r];
          else acc[e] = m * x_at(w * (NB / kCW) + lane / ST::LPR + ST::GR * r) + acc[e];
        }
      }
    }
    __syncwarp();
    if constexpr (!COLTYPE) {
      const T s = multi_group_sum<32, kTilePacks>(acc, lane);
      const T mine = __shfl_sync(0xffffffffu, s, (lane % kTilePacks) * (32 / kTilePacks));
      if (lane / kTilePacks == w) out = mine;
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
template <typename T, bool COLTYPE, bool AL>
__device__ __forceinline__ unsigned solve_block(const Args<T>& p, Block<T>& b, int rank, bool early, unsigned* ticket) {
  constexpr int NB = Geo<T>::NB, V = Geo<T>::V, WPE = Words<T>::N, SPB = NB / kStrip, NEAR = Geo<T>::NEAR, W = NearRows<T, AL>::W;
  // An NB x NB tile in registers.  Row layout: a 16 x 16 thread grid, thread (rg, cg) holds rows RS rg ..
  // RS rg + RS - 1 and the columns V cg + e, NB/2 + V cg + e: two 16-byte shared-memory loads fetch its part
  // of a vector and the row sums run over 16 lanes.  (One row per four threads needs eight loads per
  // thread, and even a broadcast load occupies the load path for its 512 bytes of results: 0.55 us a
  // product.)  Column layout, for tiles of column-type views as they lie in memory: a lane holds V rows of
  // op(A), a warp NB / 8 columns, and the sums run across the warps.
  constexpr int RS = NB / 16, CP = RS / V, H = NB / 2, JT = NB / kCW, NPK = RS * CP;
  static_assert(JT == NPK, "both tile layouts give a thread the same number of packs");
  using P = Pack<T, V>;
  auto my_ticket = [&]() {
    __syncwarp();
    cluster_wait();
    return *(volatile unsigned*)ticket;
  };
  auto enter = [&]() {
    grid_dep_wait();
    grid_dep_launch();
  };
  auto draw = [&]() {
    __syncwarp();
    cluster_wait();
    if (rank == 0 && b.tid == 0) draw_ticket(p, ticket, true);
    __syncwarp();
    cluster_arrive();
  };
  if (rank >= p.K) {
    if (!early) return 0u;
    enter();
    draw();
    return my_ticket();
  }
  T* S = b.big + Smem<T>::NEAR_ELEMS;         // inversion scratch behind the near-tile ring
  const int rg = b.tid >> 4, cg = b.tid & 15;
  const int row = rg * RS + cg / (16 / RS);        // the row whose sum this lane ends up with
  const bool owner = cg % (16 / RS) == 0;

  // near tiles: the sequence (k, w), k = rank, rank + kCS, ..., w = 2 .. min(W, K - 1 - k), NEAR tiles ahead
  int nk = rank, nw = 2, nslot = 0;
  auto near_width = [&](int k) { return min(W, p.K - 1 - k); };
  auto produce = [&]() {
    while (nk < p.K && nw > near_width(nk)) nk += kCS, nw = 2;
    if (nk < p.K) {
      const int I = mem_block(p, nk + nw), J = mem_block(p, nk);
      const int li = block_len(p, I), lj = block_len(p, J);
      T* dst = b.big + (size_t)nslot * NB * NB + (size_t)b.tid * V;
      if (!AL && li == NB && lj == NB) {
        const int ru = COLTYPE ? b.warp * JT : 2 * b.warp * RS;  // a warp's packs: one stored row, or halves of two
        const T* src = p.a + ((int64_t)(COLTYPE ? J : I) * NB + ru) * p.lda + (int64_t)(COLTYPE ? I : J) * NB + b.lane;
        dst -= b.lane * (V - 1);
        __syncwarp();
#pragma unroll
        for (int m = 0; m < NPK; ++m)
#pragma unroll
          for (int e = 0; e < V; ++e) {
            const int r = COLTYPE ? m : e * 32 / H * RS + m / CP, c = COLTYPE ? e * 32 : (m % CP) * H + e * 32 % H;
            cp_async_elem<sizeof(T)>(dst + (size_t)m * kCT * V + e * 32, src + r * p.lda + c, true);
          }
      } else
#pragma unroll
      for (int m = 0; m < NPK; ++m) {
        const int r = COLTYPE ? b.warp * JT + m : rg * RS + m / CP, c = COLTYPE ? b.lane * V : (m % CP) * H + cg * V;
        const int rows = COLTYPE ? lj : li, cols = COLTYPE ? li : lj;
        const T* src = p.a + ((int64_t)(COLTYPE ? J : I) * NB + r) * p.lda + (int64_t)(COLTYPE ? I : J) * NB + c;
        if (AL && li == NB && lj == NB) cp_async16_full(dst + (size_t)m * kCT * V, src);
        else copy_pack<T, AL>(dst + (size_t)m * kCT * V, src, r < rows ? min(V, max(0, cols - c)) : 0, p.a);
      }
      ++nw;
    }
    cp_async_commit();
    nslot = nslot + 1 == NEAR ? 0 : nslot + 1;
  };

  P inv[NPK], nxt[NPK];  // inv(D_k) and A(k+1, k), in the row layout
  auto load_inverse = [&](const T* src, int pitch) {
    if (!Diag<T, COLTYPE, AL>::transposed(p.backward)) {
#pragma unroll
      for (int m = 0; m < NPK; ++m) inv[m] = *reinterpret_cast<const P*>(src + (rg * RS + m / CP) * pitch + (m % CP) * H + cg * V);
    } else {
#pragma unroll
      for (int h = 0; h < CP; ++h)
#pragma unroll
        for (int e = 0; e < V; ++e)
#pragma unroll
          for (int a = 0; a < RS; a += V) {
            const P pk = *reinterpret_cast<const P*>(src + (h * H + cg * V + e) * pitch + rg * RS + a);
#pragma unroll
            for (int u = 0; u < V; ++u) inv[(a + u) * CP + h].v[e] = pk.v[u];
          }
    }
  };
  auto load_next = [&](int k) {
    if (k + 1 >= p.K) return;
    const int I = mem_block(p, k + 1), J = mem_block(p, k);
    const int li = block_len(p, I), lj = block_len(p, J);
    const int64_t i0 = (int64_t)I * NB + rg * RS, j0 = (int64_t)J * NB + cg * V;
    if (AL && li == NB && lj == NB) {
      if constexpr (!COLTYPE) {
#pragma unroll
        for (int m = 0; m < NPK; ++m) nxt[m] = ld_nc<T, V>(p.a + (i0 + m / CP) * p.lda + j0 + (m % CP) * H);
      } else {  // packs run along op(A)'s rows: transposed on the way into the registers
#pragma unroll
        for (int h = 0; h < CP; ++h)
#pragma unroll
          for (int e = 0; e < V; ++e)
#pragma unroll
            for (int a = 0; a < RS; a += V) {
              const P pk = ld_nc<T, V>(p.a + (j0 + h * H + e) * p.lda + i0 + a);
#pragma unroll
              for (int u = 0; u < V; ++u) nxt[(a + u) * CP + h].v[e] = pk.v[u];
            }
      }
    } else {
#pragma unroll
      for (int m = 0; m < NPK; ++m)
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const int64_t i = i0 + m / CP, j = j0 + (m % CP) * H + e;
          const bool ok = i < p.n && j < p.n;
          nxt[m].v[e] = ok ? __ldg(p.a + (COLTYPE ? j * p.lda + i : i * p.lda + j)) : T(0);
        }
    }
  };
  // A(k+1, k) into L2, ahead of load_next.
  auto prefetch_next = [&](int k) {
    if (k + 1 >= p.K) return;
    const int I = mem_block(p, k + 1), J = mem_block(p, k), R = COLTYPE ? J : I, Q = COLTYPE ? I : J;
    constexpr int LINES = NB * (int)sizeof(T) / 128;  // of a stored row of the tile
    const int rows = block_len(p, R), cols = block_len(p, Q);
#pragma unroll
    for (int i = 0; i < NB * LINES / kCT; ++i) {
      const int r = (b.tid + i * kCT) / LINES, c = (b.tid + i * kCT) % LINES * (128 / (int)sizeof(T));
      if (r < rows && c < cols) prefetch_l2(p.a + ((int64_t)R * NB + r) * p.lda + (int64_t)Q * NB + c);
    }
  };
  // row `row` of (tile in the row layout) * vec
  auto product = [&](const P (&t)[NPK], const T* vec) {
    T acc[RS];
    if constexpr (sizeof(T) == 4) {  // even and odd columns side by side: packed multiply-adds
      u64 acc2[RS];
#pragma unroll
      for (int h = 0; h < CP; ++h) {
        const ulonglong2 x2 = *reinterpret_cast<const ulonglong2*>(vec + h * H + cg * V);
#pragma unroll
        for (int a = 0; a < RS; ++a) {
          const ulonglong2 m2 = *reinterpret_cast<const ulonglong2*>(&t[a * CP + h]);
          acc2[a] = fma2(m2.x, x2.x, h == 0 ? 0ull : acc2[a]);
          acc2[a] = fma2(m2.y, x2.y, acc2[a]);
        }
      }
#pragma unroll
      for (int a = 0; a < RS; ++a) acc[a] = __uint_as_float((unsigned)acc2[a]) + __uint_as_float((unsigned)(acc2[a] >> 32));
    } else {
#pragma unroll
      for (int h = 0; h < CP; ++h) {
        const P xv = *reinterpret_cast<const P*>(vec + h * H + cg * V);
#pragma unroll
        for (int e = 0; e < V; ++e)
#pragma unroll
          for (int a = 0; a < RS; ++a) acc[a] = h == 0 && e == 0 ? t[a * CP].v[0] * xv.v[0] : t[a * CP + h].v[e] * xv.v[e] + acc[a];
      }
    }
    return multi_group_sum<16, RS>(acc, b.lane);
  };

  const unsigned slots = smem_addr(b.slots);
  int rslot = 0, par = 0;  // near-tile ring position, set of cross-warp sums
  // One block row.
  // What lies between the arrival of u_1 and the departure of the next block's u_1 runs twice, the first time
  // without its effects while the row still waits for its sums: code that has not run for microseconds is
  // fetched at a third of the speed at which it executes (u_1 to u_1 0.85 us -> 0.55 us in float).
  T bk = T(0);  // this thread's element of the right-hand side
  auto solve_row = [&](int k) {
    const int I = mem_block(p, k), li = block_len(p, I);
    u64 wd[WPE];
    P cur[NPK];
    bool pub = false;
#pragma unroll 1
    for (int t = 0; t < 2; ++t) {
      const bool go = t == 1;
      if (go && b.tid < NB) {
        T r = bk;
        if (k > W) {  // the streaming blocks' part
          const u64* q = p.far + ((int64_t)k * NB + b.tid) * WPE;
          ld_gpu(q, wd);
          while (!tagged(wd, p.tag)) {
            if (!b.wt.again()) break;
            ld_gpu(q, wd);
          }
          r -= decode(wd, T(0));
        }
        // the cluster's part, the newest last
#pragma unroll 1
        for (int w = min(W, k); w >= 1; --w) {
          const unsigned q = slots + (unsigned)(((w - 1) * NB + b.tid) * WPE * 8);
          ld_slot(q, wd);
          while (!tagged(wd, (unsigned)k + 1u)) {
            if (!b.wt.again()) break;
            ld_slot(q, wd);
          }
          r -= decode(wd, T(0));
        }
        b.rs[b.tid] = r;
      }
      if (go) bar_block();
      const T xk = product(inv, b.rs);
      if (go) {
        if (owner) b.xs[row] = xk;
        bar_block();
      }
      const T u1 = product(nxt, b.xs);
      pub = go && !*b.wt.dead && k != p.debug_skip;
      encode(u1, (unsigned)k + 2u, wd);
      st_slot_if(pub && owner && k + 1 < p.K, map_remote(slots + (unsigned)(row * WPE * 8), (unsigned)((k + 1) % kCS)), wd);
      encode(xk, p.tag, wd);
      st_gpu_if(pub && owner, p.xbuf + ((int64_t)k * NB + row) * WPE, wd);
      st_val_if(pub && owner && row < li, p.x + ((int64_t)I * NB + min(row, li - 1)) * p.incx, xk);
    }
    const int wn = near_width(k);
#pragma unroll 1
    for (int w = 2; w <= wn; ++w) {
      cp_async_wait<NEAR - 1>();
      if (!AL) __syncwarp();
      const T* src = b.big + (size_t)rslot * NB * NB + (size_t)b.tid * V;
#pragma unroll
      for (int m = 0; m < NPK; ++m) cur[m] = *reinterpret_cast<const P*>(src + (size_t)m * kCT * V);
      const unsigned dst = map_remote(slots + (unsigned)((w - 1) * NB * WPE * 8), (unsigned)((k + w) % kCS));
      if constexpr (!COLTYPE) {
        encode(product(cur, b.xs), (unsigned)(k + w) + 1u, wd);
        st_slot_if(pub && owner, dst + (unsigned)(row * WPE * 8), wd);
      } else {
        P s;
#pragma unroll
        for (int e = 0; e < V; ++e) s.v[e] = T(0);
#pragma unroll
        for (int m0 = 0; m0 < JT; m0 += V) {
          const P xv = *reinterpret_cast<const P*>(b.xs + b.warp * JT + m0);
#pragma unroll
          for (int m = 0; m < V; ++m)
#pragma unroll
            for (int e = 0; e < V; ++e) s.v[e] = cur[m0 + m].v[e] * xv.v[m] + s.v[e];
        }
        T* red = b.red + (size_t)par * kCW * NB;
        par ^= 1;
        *reinterpret_cast<P*>(red + b.warp * NB + b.lane * V) = s;
        bar_block();
        if (b.tid < NB) {
          T u = T(0);
#pragma unroll
          for (int v = 0; v < kCW; ++v) u += red[v * NB + b.tid];
          encode(u, (unsigned)(k + w) + 1u, wd);
          st_slot_if(pub, dst + (unsigned)(b.tid * WPE * 8), wd);
        }
      }
      produce();
      rslot = rslot + 1 == NEAR ? 0 : rslot + 1;
    }
    if (k + kCS < p.K) prefetch_next(k + kCS);
  };

  auto load_rhs = [&](int k) {
    const int I = mem_block(p, k);
    bk = b.tid < block_len(p, I) ? p.x[((int64_t)I * NB + b.tid) * p.incx] : T(0);
  };
  auto invert = [&](int k) {
    bar_block();
    const int I = mem_block(p, k);
    if (invert_block<T>(smem_off(S), smem_off(b.red), p.unit, block_len(p, I), b.tid)) invert_again<T, COLTYPE, AL>(p, smem_off(S), I, b.tid);
  };
  auto stage = [&](int k) { Diag<T, COLTYPE, AL>::stage(p.a, p.lda, p.n, mem_block(p, k), p.backward, S, b.tid); };

  // First row: its diagonal block, then the near tiles (in front of it they kept it waiting for 1.5 us), and the ticket in
  // the meantime.
  if (early) enter();
  load_rhs(rank);
  stage(rank);
  prefetch_next(rank);
  if (early) draw();
#pragma unroll 1
  for (int i = 0; i < NEAR; ++i) produce();
  cp_async_wait<NEAR>();
  invert(rank);
  if (early) {
    if (const unsigned t = my_ticket()) return t;
  }
#pragma unroll 1
  for (int k = rank; k < p.K; k += kCS) {
    // Inverse of the diagonal block: the first row's is formed here, the others come from the streaming
    // blocks -- or are formed here after all, when the block that should deliver one has not started.
    __shared__ int s_self;
    const T* src = S;
    int pitch = Inv<T>::SP;
    if (k != rank) {
      if (b.tid == 0) {
        s_self = p.H == 0;
        if (!s_self)
          while (ld_flag(p.flags + k) != p.tag) {
            if (!has_started(p, p.H - 1 - (k - kCS) % p.H)) {
              s_self = 1;
              break;
            }
            if (!b.wt.again()) break;
          }
      }
      bar_block();
      load_rhs(k);
      if (s_self) {
        stage(k);
        cp_async_wait<0>();
        invert(k);
      } else {
        src = p.winv + (int64_t)(k - kCS) * NB * NB, pitch = NB;
      }
    }
    load_next(k);
    load_inverse(src, pitch);
    // Sums that no running block will deliver (cold path; asked late, so that blocks that start a little
    // after this one are not taken for missing).
    if (k > W && b.warp < SPB && (p.H == 0 || !has_started(p, ((k - W - 1) * SPB + b.warp) % p.H))) {
      const T s = slow_strip<T, COLTYPE>(p, k, b.warp, k - W, b.wt, b.lane);
      u64 wd[WPE];
      encode(s, p.tag, wd);
      st_gpu_if(!*b.wt.dead, p.far + ((int64_t)k * NB + b.warp * kStrip + b.lane) * WPE, wd);
    }
    solve_row(k);
  }
  cp_async_wait<0>();
  return 0u;
}

// ---- kernel --------------------------------------------------------------------------------------------
// __grid_constant__: a function that is not inlined gets the arguments by reference, and without it every thread keeps a copy
// of them in local memory and reads that in the chain (n = 9008 in double 346 us a pair of solves, so 261).
template <typename T, bool COLTYPE, bool AL>
__global__ void __launch_bounds__(kCT, 1) trsv_cluster_kernel(const __grid_constant__ Args<T> p) {
  using SM = Smem<T>;
  constexpr int NB = Geo<T>::NB, WPE = Words<T>::N;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ unsigned s_ticket;
  __shared__ int s_dead;
  Block<T> b;
  b.big = reinterpret_cast<T*>(smem_raw);
  b.red = reinterpret_cast<T*>(smem_raw + SM::BIG);
  b.slots = reinterpret_cast<u64*>(smem_raw + SM::BIG + SM::REDTM);
  b.rs = reinterpret_cast<T*>(smem_raw + SM::BIG + SM::REDTM + SM::SLOTS);
  b.xs = b.rs + NB;
  b.tid = (int)threadIdx.x, b.warp = b.tid >> 5, b.lane = b.tid & 31;
  b.wt.budget = p.wait_limit ? p.wait_limit : (1ull << 22);
  b.wt.abort_word = p.ctl + kCtlTrsvAbort;
  b.wt.device_status = p.device_status;
  b.wt.dead = &s_dead;
  const int rank = (int)cluster_rank();
  for (int i = b.tid; i < Geo<T>::W * NB * WPE; i += kCT) b.slots[i] = 0ull;  // no stale word may look like one of this call
  if (b.tid < 2 * NB) b.rs[b.tid] = T(0);
  if (b.tid == 0) s_dead = 0;
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
  if (t == 0u) t = solve_block<T, COLTYPE, AL>(p, b, rank, early, &s_ticket);
  if (t != 0u) {
    cp_async_wait<0>();
    if (t != 0xffffffffu) stream_block<T, COLTYPE, AL>(p, b, (int)(t - 1u) * kCS + rank);
  }
  cluster_sync_all();  // no block leaves while a peer may still write into its shared memory
  // the last block out leaves the control block clean (not after an abort: the caller resets)
  if (b.tid == 0 && ld_flag(p.ctl + kCtlTrsvAbort) == 0u) {
    __threadfence();
    const unsigned d = atomicAdd(p.ctl + kCtlTrsvDone, 1u);
    if (d == gridDim.x - 1) {
      p.ctl[kCtlTrsvTicket] = 0u;
      p.ctl[kCtlTrsvDone] = 0u;
    }
  }
}

// ---- host ----------------------------------------------------------------------------------------------
// Clusters of kCS blocks of this kernel that the device holds at once (cached per device; 0: none).
template <typename T, bool COLTYPE, bool AL>
static int max_clusters() {
  static int cached[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (cached[dev] == 0) {
    auto kern = trsv_cluster_kernel<T, COLTYPE, AL>;
    int n = 0;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kCS;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(kCS);
    cfg.blockDim = dim3(kCT);
    cfg.dynamicSmemBytes = Smem<T>::TOTAL;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Smem<T>::TOTAL) != cudaSuccess ||
        cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess)
      n = 0;
    (void)cudaGetLastError();
    cached[dev] = n > 0 ? n : -1;
  }
  return cached[dev] > 0 ? cached[dev] : 0;
}

template <typename T, bool COLTYPE, bool AL>
static int launch_cluster(const Launch& l, Args<T>& p, size_t tagged_bytes, bool* handled) {
  constexpr int SPB = Geo<T>::NB / kStrip;
  int room = max_clusters<T, COLTYPE, AL>() - 1;
  if (room < 0) return B2_STATUS_OK;
  const int64_t cap = knob(kKnobTrsvStreams);
  if (cap >= 0 && cap < room) room = (int)cap;
  // streaming blocks: no more than there are strips or diagonal blocks for
  const int strips = std::max(0, p.K - NearRows<T, AL>::W - 1) * SPB, want = std::max(strips, p.K - kCS);
  const int streams = std::min(room, want <= 0 ? 0 : (want + kCS - 1) / kCS);
  p.H = streams * kCS;
  if (strips > kStrips * p.H && cap != 0) return B2_STATUS_OK;  // (no streaming blocks at all: a test's choice)
  *handled = true;
  if (int st = trsv_forget_if_captured(l, tagged_bytes)) return st;
  launch_clusters(trsv_cluster_kernel<T, COLTYPE, AL>, (unsigned)((1 + streams) * kCS), (unsigned)kCS, dim3(kCT), Smem<T>::TOTAL, l.stream, p);
  return check_launch();
}

// Workspace of a solve of K block rows: published x and far sums, flags of the inverses -- what carries tags -- and the
// inverses.
template <typename T>
struct Scratch {
  size_t words, tagged, total;
  explicit Scratch(int64_t K) {
    constexpr size_t NB = Geo<T>::NB;
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    words = up((size_t)K * NB * Words<T>::N * 8);
    tagged = 2 * words + up((size_t)K * 4);
    total = tagged + (size_t)std::max<int64_t>(0, K - kCS) * NB * NB * sizeof(T);
  }
};

}  // namespace tc

size_t trsv_cluster_scratch(int64_t n, size_t elem_bytes) {
  if (elem_bytes == 4) return tc::Scratch<float>((n + tc::Geo<float>::NB - 1) / tc::Geo<float>::NB).total;
  return tc::Scratch<double>((n + tc::Geo<double>::NB - 1) / tc::Geo<double>::NB).total;
}

template <typename T>
int trsv_cluster_try(const Launch& l, bool coltype, bool backward, bool unit, int64_t n, const T* a, int64_t lda, T* xbase, int64_t incx,
                     unsigned tag, bool* handled) {
  using namespace tc;
  constexpr int NB = Geo<T>::NB;
  *handled = false;
  const int64_t K = (n + NB - 1) / NB;
  if (K > (1 << 20)) return B2_STATUS_OK;
  const Scratch<T> w(K);
  if (w.total > l.scratch_bytes) return B2_STATUS_OK;
  Args<T> p = {};
  p.a = a;
  p.lda = lda;
  p.n = n;
  p.x = xbase;
  p.incx = incx;
  p.xbuf = reinterpret_cast<u64*>(l.scratch);
  p.far = reinterpret_cast<u64*>(l.scratch + w.words);
  p.flags = reinterpret_cast<unsigned*>(l.scratch + 2 * w.words);
  p.winv = reinterpret_cast<T*>(l.scratch + w.tagged);
  p.ctl = l.ctl;
  p.K = (int)K;
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
  const bool al = aligned_to(a, 16) && lda % Geo<T>::V == 0;
  if (coltype) return al ? launch_cluster<T, true, true>(l, p, w.tagged, handled) : launch_cluster<T, true, false>(l, p, w.tagged, handled);
  return al ? launch_cluster<T, false, true>(l, p, w.tagged, handled) : launch_cluster<T, false, false>(l, p, w.tagged, handled);
}

template int trsv_cluster_try<float>(const Launch&, bool, bool, bool, int64_t, const float*, int64_t, float*, int64_t, unsigned, bool*);
template int trsv_cluster_try<double>(const Launch&, bool, bool, bool, int64_t, const double*, int64_t, double*, int64_t, unsigned, bool*);

}  // namespace b2
