// Interface between the trsv entry points and the sub-block kernel (trsv_front.cu).
#pragma once
#include "common.cuh"

namespace b2 {

// Clears the first `bytes` (a multiple of 8) of the workspace in front of a solve that is being captured into a graph; does nothing
// otherwise.  The kernels tell values of this call from older ones by a tag that is drawn when the call is made; a
// captured solve carries the same tag on every replay, and without this would take the words that the replay before it
// left for its own.
int trsv_forget_if_captured(const Launch& l, size_t bytes);

// Tries the sub-block kernel.  Returns a status; *handled is false (and nothing was launched)
// when the call does not meet the kernel's preconditions (16-byte aligned matrix, lda a
// multiple of the pack length, workspace large enough) -- the caller then uses the general
// block-row kernel.  `xbase` is the vector base per vec_base().
template <typename T>
int trsv_front_try(const Launch& l, bool coltype, bool backward, bool unit, int64_t n, const T* a, int64_t lda,
                   T* xbase, int64_t incx, unsigned tag, bool* handled);

// The cluster kernel (trsv_cluster.cu), the same way; it takes every alignment.
template <typename T>
int trsv_cluster_try(const Launch& l, bool coltype, bool backward, bool unit, int64_t n, const T* a, int64_t lda,
                     T* xbase, int64_t incx, unsigned tag, bool* handled);
size_t trsv_cluster_scratch(int64_t n, size_t elem_bytes);  // bytes of workspace (past the control block) it needs

}  // namespace b2
