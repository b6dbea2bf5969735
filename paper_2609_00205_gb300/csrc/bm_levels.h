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

// Whether the expansion along dimension dim takes a thread per line
// (gl_expand_serial) instead of a warp per line (gl_expand): lines too long for
// the scans' segments and shared memory, or so many and so short that the
// scans' work costs more than the sweeps.  The scans are bound by issue: a line
// takes about 450 + 350 E cycles of an SM in double precision (whose unit runs
// two lanes a clock) and 100 + 40 E in single, beside a line's chain of about
// 6,000 and 2,500; the sweeps by latency, about 1,350 cycles per coarse node along
// dimensions 0 and 1 and 2,500 along dimension 2, where a thread's neighbours
// are a line apart, and by 8 per line and coarse node.  Global levels of a
// transposed decomposition with the scans (but for long lines) / the sweeps /
// this rule, in us: doubles, B = 9, K = 1: 257^3 271 / 444 / 270, 2100x30x2100
// (lines of 11 coarse nodes among longer ones) 4540 / 2806 / 2808; doubles, B = 9,
// K = 2: 1800x64x64 187 / 714 / 151; floats, B = 17, K = 2: 257^3 80 / 215 / 77;
// floats, B = 9, K = 1: 2100x30x2100 2279 / 2087 / 2098.
template <typename T>
bool expand_serial(const GLevel<T>& L, int dim, int nsm) {
  const int E = line_segment(L.d[dim].c);
  if (E == 0) return true;
  const LineShape S = line_shape(L, dim);
  const int64_t lines = S.nb * S.ncol, c = L.d[dim].c, line = sizeof(T) == 8 ? 450 + 350 * E : 100 + 40 * E;
  const int64_t chain = sizeof(T) == 8 ? 6000 : 2500;
  return chain + lines * line / nsm > c * (dim == 2 ? 2500 : 1350) + lines * c * 8 / nsm;
}

// Expansion (M_f I M_c^-1) along dimension DIM, FIN as in expand_emit.  buf:
// scratch of the fine shape (used by expand_serial's last pass).
template <typename T, int DIM, int FIN>
cudaError_t level_expand(const GLevel<T>& L, const T* in, T* buf, T* fine, const T* g, T* coef, cudaStream_t s,
                         int nsm);

}  // namespace bm
