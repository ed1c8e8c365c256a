// Library-wide pieces: workspace helpers, status strings, tuning knobs, device queries.
#include <algorithm>
#include <iterator>

#include "common.cuh"
#include "trsv_front.cuh"

namespace b2 {

static int64_t g_knobs[kKnobCount] = {
    /* kKnobL1BlocksPerSm   */ 8,
    /* kKnobGemvNTileBytes  */ 64 * 1024,
    /* kKnobGemvTRows       */ 256,
    /* kKnobTriRows         */ 0,
    /* kKnobGerRows         */ 2,
    /* kKnobUsePdl          */ 1,
    /* kKnobTrsvDebugSkip   */ -1,
    /* kKnobTriWide         */ 0,
    /* kKnobTrsvPrefetchBytes */ 12 << 20,
    /* kKnobTrsvFront       */ 3,
    /* kKnobTrsvCluster     */ 0,
    /* kKnobTrsvPmFrom      */ -1,
    /* kKnobTriTile         */ 1,
    /* kKnobTriTileUnit     */ 0,
    /* kKnobNarrowBlock     */ 1,
    /* kKnobTriBulk         */ 0,
    /* kKnobTrsvStreams     */ -1,
    /* kKnobGather          */ 1,
    /* kKnobTrsvDebugLate   */ 0,
    /* kKnobTrsvShortRows   */ -1,
};

unsigned long long g_launch_count = 0;

#ifdef B2_DEBUG_BOUNDS
static int g_dbg_shrink = 0;
static void (*g_dbg_collectors[32])(unsigned long long*);
static int g_dbg_ncollectors = 0;
int dbg_shrink() { return g_dbg_shrink; }
void dbg_register_collector(void (*fn)(unsigned long long*)) {
  if (g_dbg_ncollectors < 32) g_dbg_collectors[g_dbg_ncollectors++] = fn;
}
#endif

int64_t knob(int id) { return (id >= 0 && id < kKnobCount) ? g_knobs[id] : 0; }

int sm_count() {
  static int cached[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
  if (cached[dev] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 148;
    cached[dev] = n;
  }
  return cached[dev];
}

}  // namespace b2

extern "C" {

size_t b2_workspace_min_bytes(void) { return b2::kCtlBytes + 64 * 1024; }
size_t b2_workspace_bytes(void) { return (size_t)256 << 20; }

size_t b2_workspace_query(int64_t m, int64_t n, size_t elem_bytes) {
  if (m < 0 || n < 0 || (elem_bytes != 4 && elem_bytes != 8)) return 0;
  const size_t e = elem_bytes, V = 16 / e, seg = 32 * V;  // elements of a pack; columns of a 32-pack tile
  const size_t vec = (size_t)(m > n ? m : n), sq = (size_t)(m < n ? m : n);
  auto tiles = [](size_t len, size_t of) { return (len + of - 1) / of; };
  // column sums that a tile of shifted packs leaves to its neighbour (level2.cuh, SHIFT)
  auto spill = [&](size_t cols) { return tiles(cols + V - 1, seg) * (V - 1) * e; };
  const size_t parts[] = {
      // level 2 with every split merged: one row of partials per output vector
      ((size_t)m + (size_t)n) * e + spill(vec) + 1024,
      // narrow matrices (from 2048 rows on), column sums: one partial row per block of a resident grid
      sq <= 64 * V && vec >= 2048 ? (size_t)b2::sm_count() * 4 * sq * e : 0,
      // symv, whose blocks produce row sums and column sums at once: one row of partials per column tile of 32 packs ...
      (tiles(sq + V - 1, seg) + 1) * sq * e + spill(sq) + 1024,
      // ... and, while it runs on the ring kernel, one per tile of a block row and one per block row
      (double)sq * (double)sq * e / 2 <= b2::symv_ring_bytes(e) ? (tiles(sq, seg) + tiles(sq, 128)) * sq * e + 512 : 0,
      // trsv: tagged words and inverses of the cluster kernel; one or two words per unknown for the kernels behind it
      b2::trsv_cluster_scratch((int64_t)sq, e),
      vec * 8 * (e / 4),
  };
  return b2_workspace_min_bytes() + *std::max_element(std::begin(parts), std::end(parts));
}

int b2_workspace_reset(const b2_ctx* ctx) {
  b2::Launch l;
  if (int st = b2::make_launch(ctx, &l)) return st;
  return cudaMemsetAsync(ctx->workspace, 0, b2::kCtlBytes, l.stream) == cudaSuccess ? B2_STATUS_OK
                                                                                    : B2_STATUS_LAUNCH_FAILED;
}

const char* b2_status_string(int status) {
  if (status < 0) return "invalid argument (the negated value is its 1-based position after ctx)";
  switch (status) {
    case B2_STATUS_OK: return "ok";
    case B2_STATUS_LAUNCH_FAILED: return "CUDA launch failed";
    case B2_STATUS_WORKSPACE_TOO_SMALL: return "workspace too small";
    case B2_STATUS_NOT_IMPLEMENTED: return "not implemented";
    case B2_STATUS_TIMEOUT: return "a bounded device-side wait ran out";
    case B2_STATUS_TOO_LARGE: return "problem size above the fixed limit of this entry point";
    case B2_STATUS_BAD_CONTEXT: return "bad context (NULL, or workspace NULL / not 256-byte aligned)";
    default: return "unknown status";
  }
}

int b2_debug_bounds_report(unsigned long long* out3) {
#ifdef B2_DEBUG_BOUNDS
  if (out3 == nullptr) return -1;
  if (cudaDeviceSynchronize() != cudaSuccess) return B2_STATUS_LAUNCH_FAILED;
  out3[0] = out3[1] = out3[2] = 0;
  for (int i = 0; i < b2::g_dbg_ncollectors; ++i) b2::g_dbg_collectors[i](out3);
  return B2_STATUS_OK;
#else
  (void)out3;
  return B2_STATUS_NOT_IMPLEMENTED;
#endif
}

int b2_debug_bounds_shrink(int bytes) {
#ifdef B2_DEBUG_BOUNDS
  b2::g_dbg_shrink = bytes < 0 ? 0 : bytes;
  return B2_STATUS_OK;
#else
  (void)bytes;
  return B2_STATUS_NOT_IMPLEMENTED;
#endif
}

int b2_version(void) { return 100; }

unsigned long long b2_launch_count(void) { return b2::g_launch_count; }

int b2_set_tuning(int knob_id, int64_t value) {
  if (knob_id < 0 || knob_id >= b2::kKnobCount) return -1;
  b2::g_knobs[knob_id] = value;
  return 0;
}
int64_t b2_get_tuning(int knob_id) { return b2::knob(knob_id); }

}  // extern "C"
