// Line passes of the global levels (bm_levels.cuh), per type in their own
// translation units.
#pragma once

#include "bm_adjoint.cuh"
#include "bm_global.cuh"

namespace bm {

// One restriction pass along dimension DIM (FINAL as for gl_apply, SRC as for
// gl_line; a SRC other than SRC_GRID needs line_segment of the coarse extent).
template <typename T, int DIM, int FINAL, int SRC>
cudaError_t level_lines(const GLevel<T>& L, const T* in, T* out, const T* U, const LineSrc<T>& W, cudaStream_t s,
                        int nsm);

// Expansion (M_f I M_c^-1) along dimension DIM, FIN as in expand_emit.  buf:
// scratch of the fine shape (used by lines too long for the scans).
template <typename T, int DIM, int FIN>
cudaError_t level_expand(const GLevel<T>& L, const T* in, T* buf, T* fine, const T* g, T* coef, cudaStream_t s,
                         int nsm);

}  // namespace bm
