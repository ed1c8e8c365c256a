// Building blocks of the cluster trsv kernel (trsv_cluster.cu): tagged words, bounded waits,
// thread-block cluster access, and the inversion of a diagonal block in shared memory.
#pragma once

#include <type_traits>

#include "async_copy.cuh"

namespace b2 {
namespace tc {

using u64 = unsigned long long;

constexpr int kCT = 256;       // threads of a block (eight warps: 255 registers a thread; a ninth would leave 168)
constexpr int kCW = kCT / 32;
constexpr int kInvT = 128;     // threads that invert a diagonal block
constexpr int kBarInv = 1;     // their named barrier

// NB: unknowns per block row.  V: elements of a pack.  NEAR: near tiles in flight.  W: block rows behind the
// front whose tiles the solving cluster multiplies itself -- the slack the streaming blocks have (one fewer is
// faster below 4096 unknowns and slower above, one more the other way round: 42 / 49 / 55 us at n = 3001 and
// 158 / 155 / 152 us at n = 16384 in float).
template <typename T>
struct Geo;
template <>
struct Geo<float> {
  static constexpr int NB = 128, V = 4, NEAR = 2, W = 4;
};
template <>
struct Geo<double> {
  static constexpr int NB = 64, V = 2, NEAR = 4, W = 6;
};

// ---- tagged words: {32 payload bits, 32-bit tag}, data and ready flag in one store --------------
template <typename T>
struct Words {
  static constexpr int N = sizeof(T) / 4;
};
__device__ __forceinline__ void encode(float v, unsigned tag, u64 (&w)[1]) { w[0] = ((u64)tag << 32) | __float_as_uint(v); }
__device__ __forceinline__ void encode(double v, unsigned tag, u64 (&w)[2]) {
  const u64 b = (u64)__double_as_longlong(v);
  w[0] = ((u64)tag << 32) | (b & 0xffffffffull);
  w[1] = ((u64)tag << 32) | (b >> 32);
}
__device__ __forceinline__ float decode(const u64* w, float) { return __uint_as_float((unsigned)w[0]); }
__device__ __forceinline__ double decode(const u64* w, double) {
  return __longlong_as_double((long long)(((u64)(unsigned)w[1] << 32) | (unsigned)w[0]));
}
__device__ __forceinline__ bool tagged(const u64 (&w)[1], unsigned tag) { return (unsigned)(w[0] >> 32) == tag; }
__device__ __forceinline__ bool tagged(const u64 (&w)[2], unsigned tag) {
  return (unsigned)(w[0] >> 32) == tag && (unsigned)(w[1] >> 32) == tag;
}

// One value's words: global memory (another block of the grid writes them) and shared memory
// (another block of this cluster does).
__device__ __forceinline__ void ld_gpu(const u64* p, u64 (&w)[1]) {
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w[0]) : "l"(p) : "memory");
}
__device__ __forceinline__ void ld_gpu(const u64* p, u64 (&w)[2]) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0,%1}, [%2];" : "=l"(w[0]), "=l"(w[1]) : "l"(p) : "memory");
}
__device__ __forceinline__ void ld_slot(unsigned saddr, u64 (&w)[1]) {
  asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(w[0]) : "r"(saddr) : "memory");
}
__device__ __forceinline__ void ld_slot(unsigned saddr, u64 (&w)[2]) {
  asm volatile("ld.relaxed.cluster.shared::cta.v2.u64 {%0,%1}, [%2];" : "=l"(w[0]), "=l"(w[1]) : "r"(saddr) : "memory");
}
// Stores under a predicate instead of a branch, so that a pass that publishes nothing still fetches
// their instructions.
__device__ __forceinline__ void st_gpu_if(bool pred, u64* p, const u64 (&w)[1]) {
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %0, 0; @q st.relaxed.gpu.global.u64 [%1], %2; }" ::"r"((unsigned)pred), "l"(p),
               "l"(w[0])
               : "memory");
}
__device__ __forceinline__ void st_gpu_if(bool pred, u64* p, const u64 (&w)[2]) {
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %0, 0; @q st.relaxed.gpu.global.v2.u64 [%1], {%2,%3}; }" ::"r"((unsigned)pred),
               "l"(p), "l"(w[0]), "l"(w[1])
               : "memory");
}
__device__ __forceinline__ void st_slot_if(bool pred, unsigned raddr, const u64 (&w)[1]) {
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %0, 0; @q st.relaxed.cluster.shared::cluster.u64 [%1], %2; }" ::"r"((unsigned)pred),
               "r"(raddr), "l"(w[0])
               : "memory");
}
__device__ __forceinline__ void st_slot_if(bool pred, unsigned raddr, const u64 (&w)[2]) {
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %0, 0; @q st.relaxed.cluster.shared::cluster.v2.u64 [%1], {%2,%3}; }" ::"r"(
                   (unsigned)pred),
               "r"(raddr), "l"(w[0]), "l"(w[1])
               : "memory");
}
template <typename T>
__device__ __forceinline__ void st_val_if(bool pred, T* p, T v) {
  if (pred && !B2_GUARD(p, sizeof(T))) pred = false;
  if constexpr (sizeof(T) == 4)
    asm volatile("{ .reg .pred q; setp.ne.u32 q, %0, 0; @q st.global.f32 [%1], %2; }" ::"r"((unsigned)pred), "l"(p), "f"(v) : "memory");
  else
    asm volatile("{ .reg .pred q; setp.ne.u32 q, %0, 0; @q st.global.f64 [%1], %2; }" ::"r"((unsigned)pred), "l"(p), "d"(v) : "memory");
}
__device__ __forceinline__ unsigned ld_flag(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_flag(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// ---- thread-block cluster ------------------------------------------------------------------------
__device__ __forceinline__ void cluster_sync_all() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ unsigned map_remote(unsigned saddr, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_remote_u32(unsigned raddr, unsigned v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(raddr), "r"(v) : "memory");
}
// Block-wide barrier.  (polling loops let lanes leave at different iterations: the warp is re-converged first)
__device__ __forceinline__ void bar_block() {
  __syncwarp();
  asm volatile("barrier.sync 0;" ::: "memory");
}
__device__ __forceinline__ void bar_invert() {
  __syncwarp();
  asm volatile("barrier.sync %0, %1;" ::"n"(kBarInv), "n"(kInvT) : "memory");
}

// ---- bounded waits -------------------------------------------------------------------------------
struct Waiter {
  u64 budget;
  unsigned* abort_word;  // control block: raised by the first wait that runs out
  int* device_status;
  volatile int* dead;    // shared memory: this block has stopped waiting

  __device__ __forceinline__ void fail() {
    *dead = 1;
    atomicExch(abort_word, 1u);
    if (device_status) atomicExch(device_status, (int)B2_STATUS_TIMEOUT);
  }
  // One step of a polling loop: false when the wait is over without success.
  __device__ __forceinline__ bool again() {
    if (*dead) return false;
    if (budget == 0 || --budget == 0) {
      fail();
      return false;
    }
    if ((budget & 31) == 0 && ld_flag(abort_word) != 0u) {
      *dead = 1;
      return false;
    }
    return true;
  }
};

// Elements of a pack that exist -> shared memory, the rest zero.  AL: 16-byte copies (aligned
// matrix), else element by element.
template <typename T, bool AL>
__device__ __forceinline__ void copy_pack(T* dst, const T* src, int valid, const T* safe) {
  constexpr int V = 16 / (int)sizeof(T);
  if constexpr (AL) {
    cp_async16(dst, valid > 0 ? src : safe, valid > 0 ? valid * (int)sizeof(T) : 0);
  } else {
#pragma unroll
    for (int e = 0; e < V; ++e) cp_async_elem<sizeof(T)>(dst + e, e < valid ? src + e : safe, e < valid);
  }
}
// The whole packs of a warp off 16-byte boundaries, element by element: consecutive lanes take consecutive elements
// (dst, src: this lane's first one; the next 32 of the warp's 32 V elements lie `step` further on in global memory), so
// that a copy instruction touches one or two lines instead of the four or five of packs.  Readers wait for the warp.
template <typename T>
__device__ __forceinline__ void copy_warp(T* dst, const T* src, int64_t step) {
#pragma unroll
  for (int e = 0; e < 16 / (int)sizeof(T); ++e) cp_async_elem<sizeof(T)>(dst + e * 32, src + e * step, true);
}

// Two float multiply-adds in one instruction.
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// ---- inverse of a diagonal block -------------------------------------------------------------------
// S: NB rows of pitch SP = NB + 4 (float) / NB + 2 (double) elements holding the block in solve order,
// lower triangular; it is inverted in place by the kCT compute threads.
//   * 4 x 4 diagonal blocks by substitution, one column per thread,
//   * then, for h = 4 .. NB/2, every pair [A 0; C B] of h x h blocks gets its lower-left block
//     -inv(B) (C inv(A)): two products on register tiles, operands read as 16-byte packs.
// Bound by latency: ten short dependent steps, and code that a block executes once or twice -- hence
// one loop over the levels instead of unrolled 32 x 32 substitutions, whose straight-line code took
// 15 us of instruction fetches.
template <typename T>
struct Inv {
  static constexpr int NB = Geo<T>::NB, V = Geo<T>::V;
  static constexpr int SP = NB + V, TP = NB / 2 + V;                   // row pitches of S and Tm
  static constexpr int S_ELEMS = NB * SP, TM_ELEMS = (NB / 2) * TP;
};

template <typename T>
__device__ __forceinline__ void ld_pack(const T* p, T (&v)[16 / sizeof(T)]) {
  const Pack<T, 16 / sizeof(T)> t = *reinterpret_cast<const Pack<T, 16 / sizeof(T)>*>(p);
#pragma unroll
  for (int e = 0; e < 16 / (int)sizeof(T); ++e) v[e] = t.v[e];
}
template <typename T>
__device__ __forceinline__ void st_pack(T* p, const T (&v)[16 / sizeof(T)]) {
  Pack<T, 16 / sizeof(T)> t;
#pragma unroll
  for (int e = 0; e < 16 / (int)sizeof(T); ++e) t.v[e] = v[e];
  *reinterpret_cast<Pack<T, 16 / sizeof(T)>*>(p) = t;
}

// out[i][j] = (NEG ? - : +) sum over l in [l_lo, l_hi) of left[i][l] * right[l][j], one TI x V tile per
// thread; left, right and out are row-major in shared memory.
template <typename T, bool NEG, int TI>
__device__ __forceinline__ void tile_product(const T* left, int ldl, const T* right, int ldr, T* out, int ldo, int l_lo, int l_hi) {
  constexpr int V = 16 / (int)sizeof(T);
  T acc[TI][V];
#pragma unroll
  for (int i = 0; i < TI; ++i)
#pragma unroll
    for (int e = 0; e < V; ++e) acc[i][e] = T(0);
#pragma unroll 2
  for (int l = l_lo; l < l_hi; l += V) {
    T a[TI][V], b[V][V];
#pragma unroll
    for (int i = 0; i < TI; ++i) ld_pack(left + i * ldl + l, a[i]);
#pragma unroll
    for (int q = 0; q < V; ++q) ld_pack(right + (l + q) * ldr, b[q]);
#pragma unroll
    for (int q = 0; q < V; ++q)
#pragma unroll
      for (int i = 0; i < TI; ++i)
#pragma unroll
        for (int e = 0; e < V; ++e) acc[i][e] = a[i][q] * b[q][e] + acc[i][e];
  }
#pragma unroll
  for (int i = 0; i < TI; ++i) {
    if (NEG) {
#pragma unroll
      for (int e = 0; e < V; ++e) acc[i][e] = -acc[i][e];
    }
    st_pack(out + i * ldo, acc[i]);
  }
}

// One level for pairs of h x h blocks (h a power of two), a TI x V tile per thread; sync between the two
// products and after.  Each product skips the zero half of its triangular operand, and the tiles that are
// equally long go to the lanes of one warp: tile columns in the first product, tile rows in the second.  (The
// rows of a tile in the first product are h / TI apart, so that lanes read neighbouring rows.)
template <typename T, int TI, class Sync>
__device__ __forceinline__ void invert_level(T* S, T* Tm, int h, int tid, Sync sync) {
  constexpr int NB = Inv<T>::NB, V = Inv<T>::V, SP = Inv<T>::SP, TP = Inv<T>::TP;
  constexpr int LV = V == 4 ? 2 : 1, LT = TI == 4 ? 2 : 1;
  const int lh = 31 - __clz(h), lti = lh - LT, ltj = lh - LV, total = (NB / 2) >> lh << (lti + ltj);
  const int pr = tid >> (lti + ltj), rem = tid & ((1 << (lti + ltj)) - 1);
  const int top = pr * 2 * h, bot = top + h;
  if (tid < total) {  // Tm = C inv(A)
    const int i0 = rem & ((1 << lti) - 1), j0 = (rem >> lti) * V, is = 1 << lti;
    tile_product<T, false, TI>(S + (bot + i0) * SP + top, SP * is, S + top * SP + top + j0, SP, Tm + (pr * h + i0) * TP + j0, TP * is, j0, h);
  }
  sync();
  if (tid < total) {  // -inv(B) Tm over C
    const int j0 = (rem & ((1 << ltj) - 1)) * V, i0 = (rem >> ltj) * TI;
    tile_product<T, true, TI>(S + (bot + i0) * SP + bot, SP, Tm + (pr * h) * TP + j0, TP, S + (bot + i0) * SP + top + j0, SP, 0, i0 + TI);
  }
  sync();
}
// All levels but the last, by threads 0 .. kInvT - 1 (the diagonal counts as 1 where unit is set and from
// row nb on); the last one by all threads.
template <typename T>
__device__ __forceinline__ void invert_small(T* S, T* Tm, bool unit, int nb, int tid) {
  constexpr int NB = Inv<T>::NB, SP = Inv<T>::SP;
  T col[4];
  const int d0 = tid & ~3, lc = tid & 3;
  if (tid < NB) {
    T e[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int t = 0; t <= i; ++t) e[i][t] = (t == i && (unit || d0 + i >= nb)) ? T(1) : S[(d0 + i) * SP + d0 + t];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      T acc = i == lc ? T(1) : T(0);
#pragma unroll
      for (int t = 0; t < i; ++t) acc -= e[i][t] * col[t];
      col[i] = acc / e[i][i];
    }
  }
  bar_invert();
  if (tid < NB) {
#pragma unroll
    for (int i = 0; i < 4; ++i) S[(d0 + i) * SP + tid] = col[i];  // (exact zeros above the diagonal)
  }
  bar_invert();
#pragma unroll 1
  for (int h = 4; h < NB / 2; h *= 2) invert_level<T, 4>(S, Tm, h, tid, [] { bar_invert(); });
}
template <typename T>
__device__ __forceinline__ void invert_last(T* S, T* Tm, int tid) {
  constexpr int NB = Inv<T>::NB, V = Inv<T>::V, TI = sizeof(T) == 4 ? 4 : 2;
  static_assert((NB / 2 / TI) * (NB / 2 / V) == kCT, "one tile per thread");
  invert_level<T, TI>(S, Tm, NB / 2, tid, [] { bar_block(); });
}

// Diagonal block with memory index I.  The stored block M is lower or upper triangular; S receives the lower
// triangular one of M and its transpose, so the inverse of op(A)'s block is inv(S) or its transpose
// (`transposed`).  What lies in the unreferenced triangle is not read, but for the 4 x 4 blocks on the diagonal,
// whose upper halves are copied and then overwritten.
template <typename T, bool COLTYPE, bool AL>
struct Diag {
  static constexpr int NB = Inv<T>::NB, SP = Inv<T>::SP, V = Inv<T>::V, PPR = NB / V;
  __device__ __forceinline__ static bool transposed(bool backward) { return COLTYPE == (COLTYPE == backward); }
  __device__ __forceinline__ static void stage(const T* a, int64_t lda, int64_t n, int I, bool backward, T* S, int tid) {
    const bool stored_lower = COLTYPE == backward;
    const int64_t r0 = (int64_t)I * NB;
    const int nb = (int)min((int64_t)NB, n - r0);
    const T* src = a + r0 * lda + r0;
    if (stored_lower) {
#pragma unroll 2
      for (int idx = tid; idx < NB * PPR; idx += kCT) {
        const int r = idx / PPR, c = (idx % PPR) * V;
        copy_pack<T, AL>(S + r * SP + c, src + r * lda + c, r < nb && c <= (r | 3) ? min(V, max(0, nb - c)) : 0, a);
      }
    } else {
#pragma unroll 4
      for (int idx = tid; idx < NB * NB; idx += kCT) {  // element by element, transposed on the way
        const int c = idx / NB, r = idx % NB;           // lanes along the stored row c
        const bool ok = r < nb && c < nb && c <= (r | 3);
        cp_async_elem<sizeof(T)>(S + r * SP + c, ok ? src + c * lda + r : a, ok);
      }
    }
    cp_async_commit();
  }
};

}  // namespace tc
}  // namespace b2
