// Adjoints (transposes) of the decomposition and the recomposition.
//
// One level (Sec. II-B) maps the level grid u to (D_F, c):
//   D = (Id - I R_C) u   (zero at the all-coarse nodes),   D_F = S_F D,
//   c = R_C u + P D,      P = P_0 (x) P_1 (x) P_2,  P_k = M_c^-1 I^T M_f,
// with I the tensor interpolation from the all-coarse nodes, R_C the
// injection onto them and S_F the selection of the other nodes.  Its
// transpose, given gradients (g_D, g_c), is
//   v = S_F^T g_D + P^T g_c,   P_k^T = M_f I M_c^-1   (both mass matrices are symmetric),
//   g_u = v + R_C^T (g_c - I^T v).
// The recomposition (c - P D, then I(.) + D) is the inverse of the level; the
// transpose of that inverse, given g_u, is
//   g_c = I^T g_u,   g_D = S_F (g_u - P^T g_c).
// Both are built from two line operators applied one dimension at a time:
// "expand" (M_f I M_c^-1, coarse line to fine line) and "restrict"
// (I^T, fine line to coarse line).  The In-cache Block levels run them in
// shared memory with the compile-time tables of the forward kernels; the
// global levels run them as whole-grid passes with the plan's tables.
#pragma once

#include <atomic>

#include "bm_block.cuh"
#include "bm_global.cuh"

namespace bm {

// ---------------------------------------------------------------------------
// Block levels (uniform unit spacing, N odd, C = (N+1)/2)
// ---------------------------------------------------------------------------

// out = M_f I M_c^-1 z for one line; z[J] at in[J * stride].
template <typename T, int N>
__device__ __forceinline__ void expand_line(const BlockLevel<T, N>& tb, const T* in, int stride, T (&out)[N]) {
  constexpr int C = (N + 1) / 2;
  T y[C];
  y[0] = in[0];
#pragma unroll
  for (int i = 1; i < C; ++i) y[i] = fma(-tb.tm[i], y[i - 1], in[i * stride]);
  T z[C];
  z[C - 1] = y[C - 1] * tb.tib[C - 1];
#pragma unroll
  for (int i = C - 2; i >= 0; --i) z[i] = fma(-tb.tsup[i], z[i + 1], y[i]) * tb.tib[i];
  T w[N];
#pragma unroll
  for (int k = 0; k < N; ++k) w[k] = (k & 1) ? T(0.5) * (z[k / 2] + z[k / 2 + 1]) : z[k / 2];
  // fine mass matrix of unit spacing: diagonal 2/3 (1/3 at the ends), off-diagonal 1/6
  const T third = T(1) / T(3), sixth = T(1) / T(6);
#pragma unroll
  for (int k = 0; k < N; ++k) {
    T v = ((k == 0 || k == N - 1) ? third : T(2) * third) * w[k];
    if (k > 0) v = fma(sixth, w[k - 1], v);
    if (k < N - 1) v = fma(sixth, w[k + 1], v);
    out[k] = v;
  }
}

// r = I^T v for one line: r[J] = v[2J] + (v[2J-1] + v[2J+1]) / 2; v[k] at in[k * stride].
template <typename T, int N>
__device__ __forceinline__ void restrict_line(const T* in, int stride, T (&r)[(N + 1) / 2]) {
  constexpr int C = (N + 1) / 2;
#pragma unroll
  for (int J = 0; J < C; ++J) {
    T s = T(0);
    if (2 * J - 1 >= 0) s += in[(2 * J - 1) * stride];
    if (2 * J + 1 < N) s += in[(2 * J + 1) * stride];
    r[J] = fma(T(0.5), s, in[2 * J * stride]);
  }
}

// Expansion of a C^3 array to N^3 in shared memory: dim 0 (gc -> Y1, N C C),
// dim 1 (Y1 -> Y2, N N C); the dim-2 pass is left to the caller (`last`
// receives each (i0, i1) line's N values).
template <typename T, int N, class Last>
__device__ __forceinline__ void expand3(const T* gc, T* Y1, T* Y2, Last last) {
  constexpr int C = (N + 1) / 2;
  const auto& tb = block_tab<T, N>();
  for (int L = threadIdx.x; L < C * C; L += blockDim.x) {  // L = J1*C + J2
    T o[N];
    expand_line<T, N>(tb, gc + L, C * C, o);
#pragma unroll
    for (int i = 0; i < N; ++i) Y1[i * C * C + L] = o[i];
  }
  __syncthreads();
  for (int L = threadIdx.x; L < N * C; L += blockDim.x) {  // L = i0*C + J2
    const int i0 = L / C, j2 = L - i0 * C;
    T o[N];
    expand_line<T, N>(tb, Y1 + i0 * C * C + j2, C, o);
#pragma unroll
    for (int i = 0; i < N; ++i) Y2[(i0 * N + i) * C + j2] = o[i];
  }
  __syncthreads();
  for (int L = threadIdx.x; L < N * N; L += blockDim.x) {  // L = i0*N + i1
    T o[N];
    expand_line<T, N>(tb, Y2 + L * C, 1, o);
    last(L, o);
  }
  __syncthreads();
}

// Restriction of an N^3 array X to C^3 (out) through Y2 (N N C) and Y1 (N C C).
template <typename T, int N>
__device__ __forceinline__ void restrict3(const T* X, T* Y1, T* Y2, T* out) {
  constexpr int C = (N + 1) / 2;
  for (int L = threadIdx.x; L < N * N; L += blockDim.x) {
    T r[C];
    restrict_line<T, N>(X + L * N, 1, r);
#pragma unroll
    for (int J = 0; J < C; ++J) Y2[L * C + J] = r[J];
  }
  __syncthreads();
  for (int L = threadIdx.x; L < N * C; L += blockDim.x) {  // L = i0*C + J2
    const int i0 = L / C, j2 = L - i0 * C;
    T r[C];
    restrict_line<T, N>(Y2 + i0 * N * C + j2, C, r);
#pragma unroll
    for (int J = 0; J < C; ++J) Y1[(i0 * C + J) * C + j2] = r[J];
  }
  __syncthreads();
  for (int L = threadIdx.x; L < C * C; L += blockDim.x) {  // L = J1*C + J2
    T r[C];
    restrict_line<T, N>(Y1 + L, C * C, r);
#pragma unroll
    for (int J = 0; J < C; ++J) out[J * C * C + L] = r[J];
  }
  __syncthreads();
}

// Stream position of node k of line (i0, i1) inside its level, or -1 at an
// all-coarse node (the same order as the forward level).
template <int N>
__device__ __forceinline__ int level_pos(int L, int k) {
  constexpr int C = (N + 1) / 2;
  const int i0 = L / N, i1 = L - i0 * N;
  const bool cc = !(i0 & 1) && !(i1 & 1);
  if (cc && !(k & 1)) return -1;
  const int cc_before = ((i0 + 1) / 2) * C + ((i0 & 1) ? 0 : (i1 + 1) / 2);
  return L * N - cc_before * C + (cc ? k / 2 : k);
}

// Transposed decomposition level: gc (C^3) and the level's coefficient
// gradients (at gcoef + lvl_off) give g_u in X (N^3).  R is C^3 scratch.
template <typename T, int N>
__device__ __forceinline__ void level_adj_decompose(T* X, T* Y1, T* Y2, const T* gc, T* R, const T* gcoef,
                                                    int lvl_off) {
  constexpr int C = (N + 1) / 2;
  expand3<T, N>(gc, Y1, Y2, [&](int L, const T (&o)[N]) {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int p = level_pos<N>(L, k);
      X[L * N + k] = p >= 0 ? o[k] + gcoef[lvl_off + p] : o[k];
    }
  });
  restrict3<T, N>(X, Y1, Y2, R);
  for (int e = threadIdx.x; e < C * C * C; e += blockDim.x) {
    const int j0 = e / (C * C), r = e - j0 * C * C, j1 = r / C, j2 = r - j1 * C;
    X[((2 * j0) * N + 2 * j1) * N + 2 * j2] += gc[e] - R[e];
  }
  __syncthreads();
}

// Transposed recomposition level: X (N^3, g_u) gives gc (C^3) and the
// level's coefficient gradients (written at gcoef + lvl_off).
template <typename T, int N>
__device__ __forceinline__ void level_adj_recompose(const T* X, T* Y1, T* Y2, T* gc, T* gcoef, int lvl_off) {
  restrict3<T, N>(X, Y1, Y2, gc);
  expand3<T, N>(gc, Y1, Y2, [&](int L, const T (&o)[N]) {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int p = level_pos<N>(L, k);
      if (p >= 0) gcoef[lvl_off + p] = X[L * N + k] - o[k];
    }
  });
}

template <typename T, int N, int L, int B>
struct AdjDecLevels {  // levels L, L-1, ..., 0 (level L has N nodes)
  __device__ __forceinline__ static void run(const LevelBufs<T>& bufs, T* Y1, T* Y2, T* R, const T* gcoef) {
    level_adj_decompose<T, N>(bufs(L), Y1, Y2, bufs(L + 1), R, gcoef, lvl_offset(B, L));
    if constexpr (L > 0) AdjDecLevels<T, 2 * N - 1, L - 1, B>::run(bufs, Y1, Y2, R, gcoef);
  }
};

template <typename T, int N, int L, int K, int B>
struct AdjRecLevels {  // levels L, L+1, ..., K-1
  __device__ __forceinline__ static void run(const LevelBufs<T>& bufs, T* Y1, T* Y2, T* gcoef) {
    level_adj_recompose<T, N>(bufs(L), Y1, Y2, bufs(L + 1), gcoef, lvl_offset(B, L));
    if constexpr (L + 1 < K) AdjRecLevels<T, (N + 1) / 2, L + 1, K, B>::run(bufs, Y1, Y2, gcoef);
  }
};

template <typename T, int B, int K>
struct AdjCfg {
  using Cfg = BlockCfg<T, B, K>;
  // A (B^3), Y2 (B^2 C1), Y1 (B C1^2), cb0 (C1^3), cb1 (C2^3), R (C1^3)
  static constexpr size_t smem = sizeof(T) * (Cfg::A + Cfg::T1 + Cfg::T2 + 2 * Cfg::CB0 + Cfg::CB1);
};

// DIR 0: transposed decomposition (a.coef: coefficient gradients, a.G: block
// coarse gradients -> a.field: field gradients at the in-domain nodes).
// DIR 1: transposed recomposition (a.field -> a.coef, a.G).
template <typename T, int B, int K, int DIR>
__global__ void __launch_bounds__(BlockCfg<T, B, K>::NT_INV) block_adj_kernel(BlockArgs<T> a) {
  using Cfg = BlockCfg<T, B, K>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* A = reinterpret_cast<T*>(smem_raw);
  T* Y2 = A + Cfg::A;
  T* Y1 = Y2 + Cfg::T1;
  T* cb0 = Y1 + Cfg::T2;
  T* cb1 = cb0 + Cfg::CB0;
  T* R = cb1 + Cfg::CB1;
  LevelBufs<T> bufs{A, cb0, cb1};
  constexpr int M = Cfg::M;
  for (int64_t b = blockIdx.x; b < a.nblocks; b += gridDim.x) {
    const BlockCoord bc(b, a.nb1, a.nb2);
    T* gcoef = a.coef + b * (int64_t)Cfg::PB;
    T* g = a.G + (((int64_t)bc.b0 * M) * a.g1 + (int64_t)bc.b1 * M) * a.g2 + (int64_t)bc.b2 * M;
    T* cf = bufs(K);
    if (DIR == 0) {
      for (int e = threadIdx.x; e < M * M * M; e += blockDim.x) {
        const int j0 = e / (M * M), r = e - j0 * M * M, j1 = r / M, j2 = r - j1 * M;
        cf[e] = g[((int64_t)j0 * a.g1 + j1) * a.g2 + j2];
      }
      __syncthreads();
      AdjDecLevels<T, M * 2 - 1, K - 1, B>::run(bufs, Y1, Y2, R, gcoef);
      store_block<T, B>(BlockSpan<T, B>(a.field, a.n0, a.n1, a.n2, bc), A, a.n1, a.n2);
    } else {
      issue_block_load<T, B>(A, a.field, BlockSpan<const T, B>(a.field, a.n0, a.n1, a.n2, bc), a.n1, a.n2);
      cp_async_commit();
      cp_async_wait<0>();
      __syncthreads();
      AdjRecLevels<T, B, 0, K, B>::run(bufs, Y1, Y2, gcoef);
      for (int e = threadIdx.x; e < M * M * M; e += blockDim.x) {
        const int j0 = e / (M * M), r = e - j0 * M * M, j1 = r / M, j2 = r - j1 * M;
        g[((int64_t)j0 * a.g1 + j1) * a.g2 + j2] = cf[e];
      }
    }
    __syncthreads();
  }
}

template <typename T, int B, int K>
cudaError_t launch_adj_one(int dir, const BlockArgs<T>& a, cudaStream_t s, int nsm) {
  using Cfg = BlockCfg<T, B, K>;
  const void* fn = dir == 0 ? (const void*)block_adj_kernel<T, B, K, 0> : (const void*)block_adj_kernel<T, B, K, 1>;
  const size_t smem = AdjCfg<T, B, K>::smem;
  static std::atomic<int> cached[2][64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  int per_sm = dev < 64 ? cached[dir][dev].load() : 0;
  if (per_sm <= 0) {
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, Cfg::NT_INV, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    if (dev < 64) cached[dir][dev].store(per_sm);
  }
  int64_t grid = (int64_t)per_sm * nsm;
  if (grid > a.nblocks) grid = a.nblocks;
  if (grid < 1) return cudaSuccess;
  if (dir == 0) block_adj_kernel<T, B, K, 0><<<(unsigned)grid, Cfg::NT_INV, smem, s>>>(a);
  else block_adj_kernel<T, B, K, 1><<<(unsigned)grid, Cfg::NT_INV, smem, s>>>(a);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Global levels (physical coordinates, plan tables)
// ---------------------------------------------------------------------------

// A line pass along one dimension between a grid with n nodes on it (fine
// side) and one with c (coarse side).  Shapes as in apply_shape: lines are
// (batch b, column col); node i of the fine line is at
// fine + b*f_b + i*f_i + col*f_c, node J of the coarse line likewise.
struct LineShape {
  int64_t nb, ncol;
  int64_t f_b, f_i, f_c;
  int64_t c_b, c_i, c_c;
};

template <typename T>
LineShape line_shape(const GLevel<T>& L, int dim) {
  const ApplyShape A = apply_shape(L, dim);  // fine -> coarse restriction layout
  return LineShape{A.nb, A.ncol, A.in_b, A.in_i, A.in_c, A.out_b, A.out_j, A.out_c};
}

// What an expansion does with t = (M_f I M_c^-1 x) at a fine node: EXP_STORE
// stores it; the last (dim 2) pass of the transposed decomposition writes
// v = S_F^T g_D + t (EXP_ADD), that of the transposed recomposition the
// coefficient gradient g_u - t (EXP_COEF).
enum { EXP_STORE = 0, EXP_ADD = 1, EXP_COEF = 2 };

template <typename T, int FIN>
__device__ __forceinline__ void expand_emit_at(const GLevel<T>& L, T* fine, const T* g, T* coef, int i0, int i1, int i2,
                                               int64_t o, T t) {
  const bool cc = all_coarse(L, i0, i1, i2);
  const int64_t pos = cc ? 0 : nc_pos(L, i0, i1, i2, o);
  if (FIN == EXP_ADD) fine[o] = (cc ? T(0) : coef[pos]) + t;
  else if (!cc) coef[pos] = g[o] - t;
}
template <typename T, int FIN>
__device__ __forceinline__ void expand_emit(const GLevel<T>& L, const LineShape& S, T* fine, const T* g, T* coef,
                                            int64_t b, int64_t col, int i, T t) {
  const int64_t o = b * S.f_b + (int64_t)i * S.f_i + col * S.f_c;
  if (FIN == EXP_STORE) {
    fine[o] = t;
    return;
  }
  const int n1 = L.d[1].n, i0 = (int)(col / n1), i1 = (int)(col - (int64_t)i0 * n1);
  expand_emit_at<T, FIN>(L, fine, g, coef, i0, i1, i, o, t);
}

// fine line = M_f I M_c^-1 (coarse line), line by line along dimension DIM.
// A CTA stages 2^lsh coarse lines in shared memory (shared memory and line
// counts as for gl_line); a warp solves a line with the scans of
// line_scan_solve and interpolates it to the fine nodes, and the mass matrix is
// applied as the lines are written.  The mass matrix smooths: neighbouring
// rows' roundings that alternate, as the sweeps leave them, cancel in it, and
// the scan's independent ones do not (FP32, 21 rows: the fine line's error
// 6.77e-8 of its norm against the sweeps' 6.30e-8), so the lanes replay their
// rows from each other's results until a lane's chain of own roundings is seven
// rows or more (6.30e-8).  Bound by latency: the chain of a line
// is O(log) steps instead of the 2 c of a Thomas sweep, and a line is a warp's
// work instead of a thread's.  (Global levels of the transposed decomposition of
// 257^3 floats, B = 17, K = 2: 215 us with a thread per line, 77 with the scans.)
template <typename T, int DIM, int FIN, int E>
__global__ void __launch_bounds__(256) gl_expand(GLevel<T> L, LineShape S, const T* __restrict__ coarse,
                                                 T* __restrict__ fine, const T* __restrict__ g, T* __restrict__ coef,
                                                 const int lsh) {
  const int LT = 1 << lsh;  // lines of the CTA
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const GDim<T>& D = L.d[DIM];
  const int n = D.n, c = D.c, sn = n | 1, sc = c | 1;
  T* s_f = reinterpret_cast<T*>(smem_raw);  // [LT][sn] I M_c^-1 x
  T* s_c = s_f + LT * sn;                   // [LT][sc] x, then M_c^-1 x
  const int64_t tiles = (S.ncol + LT - 1) / LT;
  const int64_t b = blockIdx.x / tiles;
  const int64_t col0 = (blockIdx.x - b * tiles) * LT;
  const int nl = (int)(S.ncol - col0 < LT ? S.ncol - col0 : LT);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const T* x = coarse + b * S.c_b;
  if (S.c_i == 1) {
    for (int w = warp; w < nl; w += 8)
      for (int J = lane; J < c; J += 32) s_c[w * sc + J] = x[(col0 + w) * S.c_c + J];
  } else {
    for (int e = threadIdx.x; e < c * LT; e += 256) {
      const int J = e >> lsh, w = e - (J << lsh);
      if (w < nl) s_c[w * sc + J] = x[(int64_t)J * S.c_i + (col0 + w) * S.c_c];
    }
  }
  __syncthreads();
  const bool same = c == n;  // a dimension of at most two nodes is not coarsened
  if (!same) {
    for (int w = warp; w < nl; w += 8) {
      T* z = s_c + w * sc;
      line_scan_solve<T, E, E == 1 ? 6 : E == 3 ? 2 : 1>(D, z, lane);
      __syncwarp();
      for (int i = lane; i < n; i += 32) {
        const T zl = z[D.jlo[i]], zr = z[D.jhi[i]];
        s_f[w * sn + i] = D.isc[i] ? zl : fma(D.wl[i], zl, D.wr[i] * zr);
      }
    }
    __syncthreads();
  }
  auto emit = [&](int i, int w) {
    T t;
    if (same) {
      t = s_c[w * sc + i];
    } else {
      const T* y = s_f + w * sn;
      t = D.md[i] * y[i];
      if (i > 0) t = fma(D.mo[i - 1], y[i - 1], t);
      if (i + 1 < n) t = fma(D.mo[i], y[i + 1], t);
    }
    expand_emit<T, FIN>(L, S, fine, g, coef, b, col0 + w, i, t);
  };
  if (S.f_i == 1) {
    for (int w = warp; w < nl; w += 8)
      for (int i = lane; i < n; i += 32) emit(i, w);
  } else {
    for (int e = threadIdx.x; e < n * LT; e += 256) {
      const int i = e >> lsh, w = e - (i << lsh);
      if (w < nl) emit(i, w);
    }
  }
}

// The expansion by one thread per line (expand_serial): Thomas sweeps with the
// coarse values kept in the fine line's coarse slots, then the fine slots by
// interpolation, then the mass matrix with a rolling window, in place.
template <typename T>
__global__ void __launch_bounds__(256) gl_expand_serial(GDim<T> D, LineShape S, const T* __restrict__ coarse,
                                                         T* __restrict__ fine) {
  const int n = D.n, c = D.c;
  const int64_t lines = S.nb * S.ncol;
  for (int64_t line = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; line < lines;
       line += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = line / S.ncol, col = line - b * S.ncol;
    const T* x = coarse + b * S.c_b + col * S.c_c;
    T* y = fine + b * S.f_b + col * S.f_c;
    const int64_t so = S.f_i, si = S.c_i;
    if (c == n) {  // a dimension of at most two nodes is not coarsened
      for (int i = 0; i < n; ++i) y[i * so] = x[i * si];
      continue;
    }
    T yv = x[0];
    y[(int64_t)D.cidx[0] * so] = yv;
    for (int J = 1; J < c; ++J) {
      yv = fma(-D.tm[J], yv, x[J * si]);
      y[(int64_t)D.cidx[J] * so] = yv;
    }
    T z = yv * D.tib[c - 1];
    y[(int64_t)D.cidx[c - 1] * so] = z;
    for (int J = c - 2; J >= 0; --J) {
      z = fma(-D.tsup[J], z, y[(int64_t)D.cidx[J] * so]) * D.tib[J];
      y[(int64_t)D.cidx[J] * so] = z;
    }
    for (int i = 0; i < n; ++i)
      if (!D.isc[i])
        y[i * so] = fma(D.wl[i], y[(int64_t)D.cidx[D.jlo[i]] * so], D.wr[i] * y[(int64_t)D.cidx[D.jhi[i]] * so]);
    T wm = T(0), w0 = y[0];
    for (int i = 0; i < n; ++i) {
      const T wp = i + 1 < n ? y[(i + 1) * so] : T(0);
      T v = D.md[i] * w0;
      if (i > 0) v = fma(D.mo[i - 1], wm, v);
      if (i + 1 < n) v = fma(D.mo[i], wp, v);
      y[i * so] = v;
      wm = w0;
      w0 = wp;
    }
  }
}

// What gl_expand's last pass does with t as it emits it, over a grid of t: a
// thread a node, so that the grids and the coefficients are walked in order (a
// thread per line wrote and read them a line apart: 2100x30x2100 doubles, B = 9,
// K = 1, the whole gradient 15.5 ms).
template <typename T, int FIN>
__global__ void __launch_bounds__(256) gl_expand_finish(GLevel<T> L, NodeDiv nd, const T* __restrict__ t,
                                                         T* __restrict__ fine, const T* __restrict__ g,
                                                         T* __restrict__ coef) {
  const int64_t total = (int64_t)L.d[0].n * L.d[1].n * L.d[2].n;
  for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < total; o += (int64_t)gridDim.x * blockDim.x) {
    int i0, i1, i2;
    node_of(nd, o, i0, i1, i2);
    expand_emit_at<T, FIN>(L, fine, g, coef, i0, i1, i2, o, t[o]);
  }
}

// coarse = I^T fine in all three dimensions: each coarse node gathers itself
// and its fine neighbours with their interpolation weights, dimension 2
// innermost (op for op the three line passes that it stands for, which wrote
// and read two intermediate grids).  CORRECT 0 stores it; CORRECT 1 adds
// g_c - I^T v to v at the node itself (no other node's stencil reads an
// all-coarse node, so in place).
template <typename T, int CORRECT>
__global__ void __launch_bounds__(256) gl_restrict_interp(GLevel<T> L, NodeDiv cd, T* __restrict__ fine,
                                                           T* __restrict__ coarse) {
  const GDim<T>&D0 = L.d[0], &D1 = L.d[1], &D2 = L.d[2];
  const int64_t n1 = D1.n, n2 = D2.n;
  const int64_t total = (int64_t)D0.c * D1.c * D2.c;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    int j0, j1, j2;
    node_of(cd, e, j0, j1, j2);
    const int i0 = D0.cidx[j0], i1 = D1.cidx[j1], i2 = D2.cidx[j2];
    const bool l0 = i0 > 0 && !D0.isc[i0 - 1], r0 = i0 + 1 < D0.n && !D0.isc[i0 + 1];
    const bool l1 = i1 > 0 && !D1.isc[i1 - 1], r1 = i1 + 1 < D1.n && !D1.isc[i1 + 1];
    const bool l2 = i2 > 0 && !D2.isc[i2 - 1], r2 = i2 + 1 < D2.n && !D2.isc[i2 + 1];
    const T wl0 = l0 ? D0.wr[i0 - 1] : T(0), wr0 = r0 ? D0.wl[i0 + 1] : T(0);
    const T wl1 = l1 ? D1.wr[i1 - 1] : T(0), wr1 = r1 ? D1.wl[i1 + 1] : T(0);
    const T wl2 = l2 ? D2.wr[i2 - 1] : T(0), wr2 = r2 ? D2.wl[i2 + 1] : T(0);
    const int64_t u = ((int64_t)i0 * n1 + i1) * n2 + i2;
    auto line = [&](const T* x) {
      T v = x[0];
      if (l2) v = fma(wl2, x[-1], v);
      if (r2) v = fma(wr2, x[1], v);
      return v;
    };
    auto plane = [&](const T* x) {
      T v = line(x);
      if (l1) v = fma(wl1, line(x - n2), v);
      if (r1) v = fma(wr1, line(x + n2), v);
      return v;
    };
    T v = plane(fine + u);
    if (l0) v = fma(wl0, plane(fine + u - n1 * n2), v);
    if (r0) v = fma(wr0, plane(fine + u + n1 * n2), v);
    if (CORRECT) fine[u] += coarse[e] - v;
    else coarse[e] = v;
  }
}

}  // namespace bm
