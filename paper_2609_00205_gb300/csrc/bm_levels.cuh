// Launches of the line passes of the global levels (restrictions and their
// transposes): the segment length and the lines of a CTA by the level's shape.
// Instantiated by bm_levels_f32.cu and bm_levels_f64.cu, apart from the other
// kernels so that they compile side by side.
#pragma once

#include <algorithm>
#include <atomic>

#include "bm_adjoint.cuh"
#include "bm_global.cuh"
#include "bm_levels.h"
#include "bm_smem.h"

namespace bm {

// The most shared memory that lines of at most E coarse nodes a lane take: a
// full tile (128 bytes across the lines) of 2 * 32 E - 1 and 32 E nodes.
constexpr int line_smem_max(int E) { return 128 * 96 * E; }

template <typename T, int DIM, int FINAL, int SRC, int E, int LSH>
cudaError_t launch_line_tile(const GLevel<T>& L, const ApplyShape& S, const T* in, T* out, const T* U,
                             const LineSrc<T>& W, cudaStream_t s) {
  const GDim<T>& D = L.d[DIM];
  const size_t smem = line_smem<T>(D.n, D.c, LSH);
  if (line_smem_max(E) > 48 * 1024) {
    static std::atomic<unsigned> allowed{0};
    const cudaError_t e = set_smem_once(gl_line<T, DIM, FINAL, E, SRC, LSH>, line_smem_max(E), allowed);
    if (e != cudaSuccess) return e;
  }
  const int64_t ctas = S.nb * ((S.ncol + (1 << LSH) - 1) >> LSH);
  gl_line<T, DIM, FINAL, E, SRC, LSH><<<(unsigned)ctas, 256, smem, s>>>(L, S, in, out, U, W);
  return cudaGetLastError();
}
template <typename T, int DIM, int FINAL, int SRC, int E>
cudaError_t launch_line(const GLevel<T>& L, const ApplyShape& S, const T* in, T* out, const T* U, const LineSrc<T>& W,
                        cudaStream_t s, int nsm) {
  constexpr int full = line_full_shift<T>();
  if (line_tile_shift<T>(S.nb, S.ncol, nsm) == full)
    return launch_line_tile<T, DIM, FINAL, SRC, E, full>(L, S, in, out, U, W, s);
  return launch_line_tile<T, DIM, FINAL, SRC, E, full - 2>(L, S, in, out, U, W, s);
}

template <typename T, int DIM, int FINAL, int SRC>
cudaError_t level_lines(const GLevel<T>& L, const T* in, T* out, const T* U, const LineSrc<T>& W, cudaStream_t s,
                        int nsm) {
  const ApplyShape S = apply_shape(L, DIM);
  if (S.nb * S.ncol == 0) return cudaSuccess;
  switch (line_segment(L.d[DIM].c)) {
    case 1: return launch_line<T, DIM, FINAL, SRC, 1>(L, S, in, out, U, W, s, nsm);
    case 3: return launch_line<T, DIM, FINAL, SRC, 3>(L, S, in, out, U, W, s, nsm);
    case 9: return launch_line<T, DIM, FINAL, SRC, 9>(L, S, in, out, U, W, s, nsm);
    case 17: return launch_line<T, DIM, FINAL, SRC, 17>(L, S, in, out, U, W, s, nsm);
    default: break;
  }
  if (SRC != SRC_GRID) return cudaErrorInvalidValue;  // the caller's rule
  const int64_t ctas = S.nb * ((S.ncol + kApplyCols - 1) / kApplyCols);
  gl_apply<T, DIM, FINAL><<<(unsigned)ctas, 256, 0, s>>>(L, S, in, out, U);
  return cudaGetLastError();
}
template <typename T, int DIM, int FIN, int E>
cudaError_t launch_expand_line(const GLevel<T>& L, const LineShape& S, const T* in, T* fine, const T* g, T* coef,
                               cudaStream_t s, int nsm) {
  const GDim<T>& D = L.d[DIM];
  const int lsh = line_tile_shift<T>(S.nb, S.ncol, nsm);
  const size_t smem = line_smem<T>(D.n, D.c, lsh);
  if (line_smem_max(E) > 48 * 1024) {
    static std::atomic<unsigned> allowed{0};
    const cudaError_t e = set_smem_once(gl_expand<T, DIM, FIN, E>, line_smem_max(E), allowed);
    if (e != cudaSuccess) return e;
  }
  const int64_t ctas = S.nb * ((S.ncol + (1 << lsh) - 1) >> lsh);
  gl_expand<T, DIM, FIN, E><<<(unsigned)ctas, 256, smem, s>>>(L, S, in, fine, g, coef, lsh);
  return cudaGetLastError();
}

template <typename T, int DIM, int FIN>
cudaError_t level_expand(const GLevel<T>& L, const T* in, T* buf, T* fine, const T* g, T* coef, cudaStream_t s,
                         int nsm) {
  const LineShape S = line_shape(L, DIM);
  if (!expand_serial(L, DIM, nsm)) {
    switch (line_segment(L.d[DIM].c)) {
      case 1: return launch_expand_line<T, DIM, FIN, 1>(L, S, in, fine, g, coef, s, nsm);
      case 3: return launch_expand_line<T, DIM, FIN, 3>(L, S, in, fine, g, coef, s, nsm);
      case 9: return launch_expand_line<T, DIM, FIN, 9>(L, S, in, fine, g, coef, s, nsm);
      case 17: return launch_expand_line<T, DIM, FIN, 17>(L, S, in, fine, g, coef, s, nsm);
      default: return cudaErrorInvalidValue;  // the rule
    }
  }
  const int64_t cap = 8ll * nsm;
  gl_expand_serial<T><<<(unsigned)std::min<int64_t>((S.nb * S.ncol + 255) / 256, cap), 256, 0, s>>>(
      L.d[DIM], S, in, FIN == EXP_STORE ? fine : buf);
  if constexpr (FIN != EXP_STORE) {
    const int64_t nn = (int64_t)L.d[0].n * L.d[1].n * L.d[2].n;
    gl_expand_finish<T, FIN><<<(unsigned)std::min<int64_t>((nn + 255) / 256, cap), 256, 0, s>>>(L, node_div(L), buf,
                                                                                               fine, g, coef);
  }
  return cudaGetLastError();
}

#define BM_LINES(T, DIM, FINAL, SRC)                                                                        \
  template cudaError_t level_lines<T, DIM, FINAL, SRC>(const GLevel<T>&, const T*, T*, const T*, const LineSrc<T>&, \
                                                       cudaStream_t, int);
#define BM_EXPAND(T, DIM, FIN)                                                                            \
  template cudaError_t level_expand<T, DIM, FIN>(const GLevel<T>&, const T*, T*, T*, const T*, T*, cudaStream_t, int);
#define BM_LEVELS(T)                                                                                             \
  BM_LINES(T, 2, 0, SRC_GRID)                                                                                    \
  BM_LINES(T, 2, 0, SRC_CODE)                                                                                    \
  BM_LINES(T, 2, 0, SRC_COEF)                                                                                    \
  BM_LINES(T, 2, 0, SRC_DECODE)                                                                                  \
  BM_LINES(T, 2, 0, SRC_READ)                                                                                    \
  BM_LINES(T, 1, 0, SRC_GRID)                                                                                    \
  BM_LINES(T, 1, 1, SRC_GRID)                                                                                    \
  BM_LINES(T, 1, 2, SRC_GRID)                                                                                    \
  BM_LINES(T, 0, 1, SRC_GRID)                                                                                    \
  BM_LINES(T, 0, 2, SRC_GRID)                                                                                    \
  BM_EXPAND(T, 0, EXP_STORE)                                                                                     \
  BM_EXPAND(T, 1, EXP_STORE)                                                                                     \
  BM_EXPAND(T, 2, EXP_ADD)                                                                                       \
  BM_EXPAND(T, 2, EXP_COEF)

}  // namespace bm
