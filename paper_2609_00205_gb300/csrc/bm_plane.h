// Arguments and launchers of the fused block kernels of 2-D fields.
#pragma once

#include <cuda_runtime.h>

#include "bm_common.cuh"

namespace bm {

// Device tables of one in-cache level (both axes share them).
template <typename T>
struct PlaneLevel {
  const T *band, *tm, *tib, *tsup;
};

template <typename T>
struct PlaneArgs {
  T* field;  // forward: input (read); inverse: output (written)
  int64_t e0, e1, st0, st1;  // extents and element strides of the field's two axes
  int nb1;                   // blocks along the second axis
  int64_t nblocks;
  T* G;  // gathered block-coarse grid
  int64_t gs0, gs1;
  uint16_t* sym;
  int32_t* esc;
  const uint8_t* tier;  // per block tier or null
  const T* rq;          // forward: 1/q per [tier*K + level]
  const double* q;      // inverse: q per [tier*K + level]
  int radius, ntiers;
  Scalars* sc;
  PlaneLevel<T> lev[4];
};

// Whether the fused kernels take a field's in-cache levels: two axes longer
// than 1 and blocks of 9 or 17 nodes (other block sizes, 1-D fields and the
// full-precision coefficients take the whole-grid passes).
inline bool plane_fused(bool two_axes, int B, int K) {
  return two_axes && ((B == 9 && K <= 3) || (B == 17 && K <= 4));
}

// dir 0 = decompose and quantise, 1 = dequantise and recompose.
cudaError_t launch_plane(int dir, int B, int K, const PlaneArgs<float>& a, cudaStream_t s, int nsm);
cudaError_t launch_plane(int dir, int B, int K, const PlaneArgs<double>& a, cudaStream_t s, int nsm);

}  // namespace bm
