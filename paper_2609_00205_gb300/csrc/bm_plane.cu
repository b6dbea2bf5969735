// Fused In-cache Block kernels of coded 2-D fields (3-D fields with one extent
// of 1 among them) with blocks of 9 or 17 nodes per edge: a CTA takes NB
// consecutive blocks through all K levels in shared memory, a thread per line.
// As whole-grid passes (gather, then per level coefficients, two line passes
// and the coarse correction, scatter) the blocks of a 1535x2049 field took
// 0.322 ms in ten launches, bound by latency and by index arithmetic; fused,
// 0.031 ms, bound by issue (a tile of 289 nodes is little work between barriers).
//
// The arithmetic is that of the whole-grid kernels (gl_fwd_detail, gl_line,
// gl_ident0, gl_inv_dequant, gl_inv_interp), operation for operation, so the
// streams are the same bytes: gl_line evaluates the two Thomas recurrences as
// warp scans of affine maps, one row per lane; here a thread runs the same
// scan over its registers, and the maps' products, which do not depend on the
// data, come from a table built once per CTA.
#include "bm_internal.h"
#include "bm_plane.h"

#include <atomic>

namespace bm {
namespace {

constexpr int pl_n(int B, int l) { return l == 0 ? B : (pl_n(B, l - 1) + 1) / 2; }
constexpr int pl_per_block(int B, int K) {
  return K == 0 ? 0 : B * B - ((B + 1) / 2) * ((B + 1) / 2) + pl_per_block((B + 1) / 2, K - 1);
}
constexpr int pl_offset(int B, int l) { return pl_per_block(B, l); }

// A level's operators on lines of N = 2C - 1 nodes: the band of I^T M_f, the
// Thomas factors of M_c, and the multipliers of the scans' stages (offsets 1,
// 2, 4, 8).
template <typename T, int C>
struct LineTab {
  static constexpr int S = C > 8 ? 4 : C > 4 ? 3 : C > 2 ? 2 : 1;
  T band[5 * C], tm[C], tib[C], tsup[C], fm[S][C], bm[S][C];
};

template <typename T, int C>
__device__ void build_tab(LineTab<T, C>& t, const PlaneLevel<T>& L) {  // one thread
  using LT = LineTab<T, C>;
  for (int i = 0; i < 5 * C; ++i) t.band[i] = L.band[i];
  for (int J = 0; J < C; ++J) {
    t.tm[J] = L.tm[J];
    t.tib[J] = L.tib[J];
    t.tsup[J] = L.tsup[J];
    t.fm[0][J] = -t.tm[J];
    t.bm[0][J] = -t.tsup[J] * t.tib[J];
  }
  for (int s = 0; s + 1 < LT::S; ++s)
    for (int J = 0; J < C; ++J) {
      const int o = 1 << s;
      t.fm[s + 1][J] = J >= o ? t.fm[s][J] * t.fm[s][J - o] : t.fm[s][J];
      t.bm[s + 1][J] = J + o < C ? t.bm[s][J] * t.bm[s][J + o] : t.bm[s][J];
    }
}

// A product of its own rounding (not contracted with an addition that follows).
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// z = M_c^-1 I^T M_f d of one line.
template <typename T, int N>
__device__ __forceinline__ void line_solve(const LineTab<T, (N + 1) / 2>& t, const T (&d)[N], T (&z)[(N + 1) / 2]) {
  constexpr int C = (N + 1) / 2;
  T r[C], a[C];
#pragma unroll
  for (int J = 0; J < C; ++J) {
    T v = T(0);
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      const int col = (J ? 2 * J - 2 : 0) + m;
      if (col <= 2 * J + 2 && col < N) v = fma(t.band[5 * J + m], d[col], v);
    }
    r[J] = v;
    a[J] = v;
  }
#pragma unroll
  for (int s = 0; s < LineTab<T, C>::S; ++s)
#pragma unroll
    for (int J = C - 1; J >= (1 << s); --J) a[J] = fma(t.fm[s][J], a[J - (1 << s)], a[J]);
  T y[C];
#pragma unroll
  for (int J = 0; J < C; ++J) y[J] = fma(-t.tm[J], J ? a[J - 1] : T(0), r[J]);
#pragma unroll
  for (int J = 0; J < C; ++J) a[J] = y[J] * t.tib[J];
#pragma unroll
  for (int s = 0; s < LineTab<T, C>::S; ++s)
#pragma unroll
    for (int J = 0; J + (1 << s) < C; ++J) a[J] = fma(t.bm[s][J], a[J + (1 << s)], a[J]);
#pragma unroll
  for (int J = 0; J < C; ++J) z[J] = mul_rn(fma(-t.tsup[J], J + 1 < C ? a[J + 1] : T(0), y[J]), t.tib[J]);
}

// The interpolant along a row (i1) of N nodes from the coarse rows ra and rb
// (elements st apart), weights w1l and w1r (1, 0 on a coarse row).
template <typename T, int N>
__device__ __forceinline__ void interp_row(const T* ra, const T* rb, const int st, const T w1l, const T w1r,
                                           T (&e)[N]) {
  constexpr int C = (N + 1) / 2;
  T va[C], vb[C];
#pragma unroll
  for (int J = 0; J < C; ++J) {
    va[J] = ra[st * J];
    vb[J] = rb[st * J];
  }
#pragma unroll
  for (int k = 0; k < N; ++k) {
    if (k & 1)
      e[k] = fma(w1l, fma(T(0.5), va[k / 2], T(0.5) * va[k / 2 + 1]),
                 w1r * fma(T(0.5), vb[k / 2], T(0.5) * vb[k / 2 + 1]));
    else e[k] = fma(w1l, va[k / 2], w1r * vb[k / 2]);
  }
}

// In-level position of node (i1, k) of a block (row-major, all-coarse nodes
// left out).
template <int N>
__device__ __forceinline__ int row_base(int i1) {
  return i1 * N - ((i1 + 1) / 2) * ((N + 1) / 2);
}

template <typename T, int B, int K>
struct PlaneCfg {
  static constexpr int NT = 128, NB = NT / B;  // blocks: a line of the first pass per thread
  static constexpr int C1 = (B + 1) / 2, C2 = (C1 + 1) / 2, M = pl_n(B, K), PB = pl_per_block(B, K);
  static constexpr int X = B * B, T1 = C1 * B, CB0 = C1 * C1, CB1 = C2 * C2;
  static constexpr int buf_size(int j) { return j == 0 ? X : (j & 1) ? CB0 : CB1; }
};

template <typename T, int B, int K>
struct PlaneSmem {
  using Cfg = PlaneCfg<T, B, K>;
  T X[Cfg::NB * Cfg::X], T1[Cfg::NB * Cfg::T1], cb0[Cfg::NB * Cfg::CB0], cb1[Cfg::NB * Cfg::CB1];
  LineTab<T, (B + 1) / 2> t0;
  LineTab<T, (pl_n(B, 1) + 1) / 2> t1;
  LineTab<T, pl_n(B, 2) >= 3 ? (pl_n(B, 2) + 1) / 2 : 2> t2;
  LineTab<T, pl_n(B, 3) >= 3 ? (pl_n(B, 3) + 1) / 2 : 2> t3;
  T q[Cfg::NB * K];
  alignas(16) int32_t code[Cfg::NB * Cfg::PB];  // forward: symbols (16 bits each)
  __device__ __forceinline__ T* buf(int j) { return j == 0 ? X : (j & 1) ? cb0 : cb1; }
  template <int L>
  __device__ __forceinline__ auto& tab() {
    if constexpr (L == 0) return t0;
    else if constexpr (L == 1) return t1;
    else if constexpr (L == 2) return t2;
    else return t3;
  }
  __device__ void build(const PlaneArgs<T>& a) {
    if (threadIdx.x == 0) build_tab(t0, a.lev[0]);
    if (K > 1 && threadIdx.x == 32) build_tab(t1, a.lev[1]);
    if constexpr (K > 2) if (threadIdx.x == 64) build_tab(t2, a.lev[2]);
    if constexpr (K > 3) if (threadIdx.x == 96) build_tab(t3, a.lev[3]);
  }
};

template <typename T, int B, int K, int L>
__device__ __forceinline__ void plane_fwd_levels(PlaneSmem<T, B, K>& S, int32_t* esc, const unsigned dict,
                                                 const int radius, const int nv, bool& ovf) {
  using Cfg = PlaneCfg<T, B, K>;
  constexpr int N = pl_n(B, L), C = (N + 1) / 2;
  T* const X = S.buf(L);
  T* const out = S.buf(L + 1);
  constexpr int XS = Cfg::buf_size(L), OS = Cfg::buf_size(L + 1);
  const LineTab<T, C>& tb = S.template tab<L>();
  uint16_t* const stage = reinterpret_cast<uint16_t*>(S.code);
  for (int I = threadIdx.x; I < nv * N; I += Cfg::NT) {  // along the last dimension
    const int blk = I / N, i1 = I - blk * N;
    const bool odd = i1 & 1;
    const T* x = X + blk * XS;
    const T* ra = x + (odd ? i1 - 1 : i1) * N;
    const T* rb = x + (odd ? i1 + 1 : i1) * N;
    T d[N];
    interp_row<T, N>(ra, rb, 2, odd ? T(0.5) : T(1), odd ? T(0.5) : T(0), d);
#pragma unroll
    for (int k = 0; k < N; ++k) d[k] = x[i1 * N + k] - d[k];
    if (!odd) {
#pragma unroll
      for (int J = 0; J < C; ++J) out[blk * OS + (i1 / 2) * C + J] = ra[2 * J];
    }
    const int base = blk * Cfg::PB + pl_offset(B, L) + row_base<N>(i1);
    const T rq = S.q[blk * K + L];
#pragma unroll
    for (int k = 0; k < N; ++k) {
      if (odd || (k & 1)) {
        const int pos = base + (odd ? k : k / 2);
        const int code = quantize(d[k], rq, ovf);
        const unsigned u = (unsigned)(code + radius);
        const bool in = u - 1u < dict - 1u;
        stage[pos] = (uint16_t)(in ? u : 0u);
        if (!in) esc[pos] = code;
      }
    }
    T z[C];
    line_solve<T, N>(tb, d, z);
#pragma unroll
    for (int J = 0; J < C; ++J) S.T1[blk * Cfg::T1 + J * N + i1] = z[J];
  }
  __syncthreads();
  for (int I = threadIdx.x; I < nv * C; I += Cfg::NT) {  // along the first
    const int blk = I / C, j2 = I - blk * C;
    T d[N], z[C];
#pragma unroll
    for (int i = 0; i < N; ++i) d[i] = S.T1[blk * Cfg::T1 + j2 * N + i];
    line_solve<T, N>(tb, d, z);
#pragma unroll
    for (int J = 0; J < C; ++J) out[blk * OS + J * C + j2] += z[J];
  }
  __syncthreads();
  if constexpr (L + 1 < K) plane_fwd_levels<T, B, K, L + 1>(S, esc, dict, radius, nv, ovf);
}

// Elements of a group's blocks: between shared memory (blk, k1, k2) and a grid
// of blocks of edge E (strides st0, st1).
template <int E, class F>
__device__ __forceinline__ void for_nodes(int64_t b0, int nv, int nb1, int nt, F f) {
  for (int I = threadIdx.x; I < nv * E * E; I += nt) {
    const int blk = I / (E * E), r = I - blk * (E * E), k1 = r / E, k2 = r - k1 * E;
    const unsigned b = (unsigned)(b0 + blk), c0 = b / (unsigned)nb1, c1 = b - c0 * (unsigned)nb1;
    f(I, (int64_t)c0 * E + k1, (int64_t)c1 * E + k2);
  }
}

template <typename T, int B, int K>
__global__ void __launch_bounds__(128, 5) plane_fwd_kernel(PlaneArgs<T> a) {
  using Cfg = PlaneCfg<T, B, K>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PlaneSmem<T, B, K>& S = *reinterpret_cast<PlaneSmem<T, B, K>*>(smem_raw);
  S.build(a);
  bool ovf = false;
  const unsigned dict = 2u * (unsigned)a.radius;
  for (int64_t b = (int64_t)blockIdx.x * Cfg::NB; b < a.nblocks; b += (int64_t)gridDim.x * Cfg::NB) {
    const int nv = (int)(a.nblocks - b < Cfg::NB ? a.nblocks - b : Cfg::NB);
    for_nodes<B>(b, nv, a.nb1, Cfg::NT, [&](int I, int64_t c0, int64_t c1) {
      S.X[I] = c0 < a.e0 && c1 < a.e1 ? a.field[c0 * a.st0 + c1 * a.st1] : T(0);
    });
    for (int i = threadIdx.x; i < nv * K; i += Cfg::NT) {
      const int blk = i / K, tier = a.tier ? a.tier[b + blk] : 0;
      S.q[i] = __ldcg(a.rq + tier * K + (i - blk * K));
    }
    __syncthreads();
    const int64_t sb = b * (int64_t)Cfg::PB;
    plane_fwd_levels<T, B, K, 0>(S, a.esc + sb, dict, a.radius, nv, ovf);
    const T* cf = S.buf(K);
    for_nodes<Cfg::M>(b, nv, a.nb1, Cfg::NT, [&](int I, int64_t c0, int64_t c1) {
      const int blk = I / (Cfg::M * Cfg::M);
      a.G[c0 * a.gs0 + c1 * a.gs1] = cf[blk * Cfg::buf_size(K) + (I - blk * (Cfg::M * Cfg::M))];
    });
    const uint16_t* stage = reinterpret_cast<const uint16_t*>(S.code);
    if ((sb & 1) == 0) {  // pairs of symbols
      unsigned* dst = reinterpret_cast<unsigned*>(a.sym + sb);
      for (int i = threadIdx.x; i < nv * Cfg::PB / 2; i += Cfg::NT) dst[i] = reinterpret_cast<const unsigned*>(stage)[i];
      if (threadIdx.x == 0 && ((nv * Cfg::PB) & 1)) a.sym[sb + nv * Cfg::PB - 1] = stage[nv * Cfg::PB - 1];
    } else {
      for (int i = threadIdx.x; i < nv * Cfg::PB; i += Cfg::NT) a.sym[sb + i] = stage[i];
    }
    __syncthreads();
  }
  if (ovf) atomicOr(&a.sc->status, ST_OVERFLOW);
}

template <typename T, int B, int K, int L>
__device__ __forceinline__ void plane_inv_levels(PlaneSmem<T, B, K>& S, const int nv) {
  using Cfg = PlaneCfg<T, B, K>;
  constexpr int N = pl_n(B, L), C = (N + 1) / 2;
  T* const X = S.buf(L);
  T* const cin = S.buf(L + 1);
  constexpr int XS = Cfg::buf_size(L), CS = Cfg::buf_size(L + 1);
  const LineTab<T, C>& tb = S.template tab<L>();
  for (int I = threadIdx.x; I < nv * N; I += Cfg::NT) {
    const int blk = I / N, i1 = I - blk * N;
    const bool odd = i1 & 1;
    T* x = X + blk * XS + i1 * N;
    const int base = blk * Cfg::PB + pl_offset(B, L) + row_base<N>(i1);
    const T q = S.q[blk * K + L];
    T d[N], z[C];
#pragma unroll
    for (int k = 0; k < N; ++k) {
      d[k] = odd || (k & 1) ? dequant(S.code[base + (odd ? k : k / 2)], q) : T(0);
      x[k] = d[k];
    }
    line_solve<T, N>(tb, d, z);
#pragma unroll
    for (int J = 0; J < C; ++J) S.T1[blk * Cfg::T1 + J * N + i1] = z[J];
  }
  __syncthreads();
  for (int I = threadIdx.x; I < nv * C; I += Cfg::NT) {
    const int blk = I / C, j2 = I - blk * C;
    T d[N], z[C];
#pragma unroll
    for (int i = 0; i < N; ++i) d[i] = S.T1[blk * Cfg::T1 + j2 * N + i];
    line_solve<T, N>(tb, d, z);
#pragma unroll
    for (int J = 0; J < C; ++J) cin[blk * CS + J * C + j2] -= z[J];
  }
  __syncthreads();
  for (int I = threadIdx.x; I < nv * N; I += Cfg::NT) {
    const int blk = I / N, i1 = I - blk * N;
    const bool odd = i1 & 1;
    T* x = X + blk * XS + i1 * N;
    const T* c = cin + blk * CS;
    T e[N];
    interp_row<T, N>(c + (i1 >> 1) * C, c + ((i1 + 1) >> 1) * C, 1, odd ? T(0.5) : T(1), odd ? T(0.5) : T(0), e);
#pragma unroll
    for (int k = 0; k < N; ++k) x[k] = e[k] + x[k];
  }
  __syncthreads();
  if constexpr (L > 0) plane_inv_levels<T, B, K, L - 1>(S, nv);
}

template <typename T, int B, int K>
__global__ void __launch_bounds__(128, 5) plane_inv_kernel(PlaneArgs<T> a) {
  using Cfg = PlaneCfg<T, B, K>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PlaneSmem<T, B, K>& S = *reinterpret_cast<PlaneSmem<T, B, K>*>(smem_raw);
  S.build(a);
  for (int64_t b = (int64_t)blockIdx.x * Cfg::NB; b < a.nblocks; b += (int64_t)gridDim.x * Cfg::NB) {
    const int nv = (int)(a.nblocks - b < Cfg::NB ? a.nblocks - b : Cfg::NB);
    const int64_t sb = b * (int64_t)Cfg::PB;
    for (int i = threadIdx.x; i < nv * Cfg::PB; i += Cfg::NT) {
      const int s = (int)a.sym[sb + i];
      S.code[i] = s ? s - a.radius : a.esc[sb + i];
    }
    for (int i = threadIdx.x; i < nv * K; i += Cfg::NT) {
      const int blk = i / K;
      int tier = a.tier ? a.tier[b + blk] : 0;
      if (tier >= a.ntiers) {  // corrupt stream: keep the q reads inside the table
        if (a.sc) atomicOr(&a.sc->status, ST_CORRUPT);
        tier = 0;
      }
      S.q[i] = (T)a.q[tier * K + (i - blk * K)];
    }
    T* cf = S.buf(K);
    for_nodes<Cfg::M>(b, nv, a.nb1, Cfg::NT, [&](int I, int64_t c0, int64_t c1) {
      const int blk = I / (Cfg::M * Cfg::M);
      cf[blk * Cfg::buf_size(K) + (I - blk * (Cfg::M * Cfg::M))] = a.G[c0 * a.gs0 + c1 * a.gs1];
    });
    __syncthreads();
    plane_inv_levels<T, B, K, K - 1>(S, nv);
    for_nodes<B>(b, nv, a.nb1, Cfg::NT, [&](int I, int64_t c0, int64_t c1) {
      if (c0 < a.e0 && c1 < a.e1) a.field[c0 * a.st0 + c1 * a.st1] = S.X[I];
    });
    __syncthreads();
  }
}

template <typename T, int B, int K>
cudaError_t launch_k(int dir, const PlaneArgs<T>& a, cudaStream_t s, int nsm) {
  const void* fn = dir == 0 ? (const void*)plane_fwd_kernel<T, B, K> : (const void*)plane_inv_kernel<T, B, K>;
  constexpr size_t smem = sizeof(PlaneSmem<T, B, K>);
  static_assert(smem <= 100 * 1024, "two CTAs per SM at least");
  // shared-memory attribute and occupancy, once per device and direction
  static std::atomic<int> cached[2][64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  int per_sm = dev < 64 ? cached[dir][dev].load() : 0;
  if (per_sm <= 0) {
    if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, 128, smem)) != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    if (dev < 64) cached[dir][dev].store(per_sm);
  }
  const int64_t groups = (a.nblocks + PlaneCfg<T, B, K>::NB - 1) / PlaneCfg<T, B, K>::NB;
  const int64_t grid = groups < (int64_t)per_sm * nsm ? groups : (int64_t)per_sm * nsm;
  if (grid < 1) return cudaSuccess;
  if (dir == 0) plane_fwd_kernel<T, B, K><<<(unsigned)grid, 128, smem, s>>>(a);
  else plane_inv_kernel<T, B, K><<<(unsigned)grid, 128, smem, s>>>(a);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_t(int dir, int B, int K, const PlaneArgs<T>& a, cudaStream_t s, int nsm) {
  if (B == 9) {
    if (K == 1) return launch_k<T, 9, 1>(dir, a, s, nsm);
    if (K == 2) return launch_k<T, 9, 2>(dir, a, s, nsm);
    if (K == 3) return launch_k<T, 9, 3>(dir, a, s, nsm);
  } else if (B == 17) {
    if (K == 1) return launch_k<T, 17, 1>(dir, a, s, nsm);
    if (K == 2) return launch_k<T, 17, 2>(dir, a, s, nsm);
    if (K == 3) return launch_k<T, 17, 3>(dir, a, s, nsm);
    if (K == 4) return launch_k<T, 17, 4>(dir, a, s, nsm);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_plane(int dir, int B, int K, const PlaneArgs<float>& a, cudaStream_t s, int nsm) {
  return launch_t(dir, B, K, a, s, nsm);
}
cudaError_t launch_plane(int dir, int B, int K, const PlaneArgs<double>& a, cudaStream_t s, int nsm) {
  return launch_t(dir, B, K, a, s, nsm);
}

}  // namespace bm
