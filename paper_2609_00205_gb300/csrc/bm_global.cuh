// Global MGARD levels on the gathered block-coarse grid G (Sec. III-B hybrid
// hierarchy: L local levels, then M whole-grid levels).  Each level is a
// handful of whole-grid passes: coefficients, three restriction passes (one
// per dimension, shrinking it: the band product I^T M_f and the tridiagonal
// solve with M_c of that dimension) and the coarse correction; the inverse
// runs them backwards.
// Node coordinates are physical (block offset plus the node's in-block
// coordinate), so every per-dimension operator comes from a host-built table.
#pragma once

#include "bm_common.cuh"

namespace bm {

template <typename T>
struct GDim {
  int n, c;
  const int* cidx;      // [c] fine index of coarse node J
  const int* jlo;       // [n] coarse index of the left interpolation node (= J at coarse nodes)
  const int* jhi;       // [n] right node
  const T* wl;          // [n] interpolation weights (1, 0 at coarse nodes)
  const T* wr;
  const int* cb;        // [n] number of coarse indices below i
  const uint8_t* isc;   // [n] 1 at coarse nodes
  const T* P;           // [c x n] row-major projection M_c^{-1} I^T M_f
  const int* f0;        // [c] first fine column of row J of I^T M_f
  const T* band;        // [5c] row J of I^T M_f over fine columns f0[J] .. f0[J]+4
  const T* tm;          // [c] Thomas factors of M_c: y_J = r_J - tm_J y_{J-1},
  const T* tib;         //     z_J = (y_J - tsup_J z_{J+1}) tib_J
  const T* tsup;
  const T* md;          // [n] diagonal of M_f
  const T* mo;          // [n] mo[i] = M_f(i, i+1)
  int ident;            // 1: the identity of n nodes (c = n); the tables above are not used
};

// Index tables of a dimension, the identity's computed in place.
template <typename T> __device__ __forceinline__ int g_cidx(const GDim<T>& D, int i) { return D.ident ? i : D.cidx[i]; }
template <typename T> __device__ __forceinline__ int g_jlo(const GDim<T>& D, int i) { return D.ident ? i : D.jlo[i]; }
template <typename T> __device__ __forceinline__ int g_jhi(const GDim<T>& D, int i) { return D.ident ? i : D.jhi[i]; }
template <typename T> __device__ __forceinline__ T g_wl(const GDim<T>& D, int i) { return D.ident ? T(1) : D.wl[i]; }
template <typename T> __device__ __forceinline__ T g_wr(const GDim<T>& D, int i) { return D.ident ? T(0) : D.wr[i]; }
template <typename T> __device__ __forceinline__ int g_cb(const GDim<T>& D, int i) { return D.ident ? i : D.cb[i]; }
template <typename T> __device__ __forceinline__ bool g_isc(const GDim<T>& D, int i) { return D.ident || D.isc[i]; }

template <typename T>
struct GLevel {
  GDim<T> d[3];
  int64_t sym_off;    // first symbol of the level in the stream order
  int64_t blk_extra;  // added per index of dimension 0: 0 for global levels; for the in-cache levels
                      // of the block-major grid, the symbols of a block's other levels (block-major order)
  // Blocked levels (the in-cache levels of the padded grid of a round's
  // blocks, block-diagonal operators): coefficients are stored block by
  // block, bpb symbols per block, each block's level row-major over its own
  // non-coarse nodes; be / bce: a block's extent and coarse count per
  // dimension, bnb: blocks per dimension.  bmode = 0 otherwise.
  int bmode;
  int be[3], bce[3], bnb[3];
  int64_t bpb;
};

// Block (row-major over the block grid) of a node of a blocked level.
template <typename T>
__device__ __forceinline__ int64_t blk_of(const GLevel<T>& L, int i0, int i1, int i2) {
  return ((int64_t)(i0 / L.be[0]) * L.bnb[1] + i1 / L.be[1]) * L.bnb[2] + i2 / L.be[2];
}

// Stream position of a non-coarse node of a blocked level.
template <typename T>
__device__ __forceinline__ int64_t blk_pos(const GLevel<T>& L, int i0, int i1, int i2) {
  const int b0 = i0 / L.be[0], b1 = i1 / L.be[1], b2 = i2 / L.be[2];
  const int k0 = i0 - b0 * L.be[0], k1 = i1 - b1 * L.be[1], k2 = i2 - b2 * L.be[2];
  // coarse nodes of the block before the node: from the line tables, whose
  // coarse counts run over the whole padded line
  const int64_t c0 = L.d[0].cb[i0] - (int64_t)b0 * L.bce[0];
  const int64_t c1 = L.d[1].cb[i1] - (int64_t)b1 * L.bce[1];
  const int64_t c2 = L.d[2].cb[i2] - (int64_t)b2 * L.bce[2];
  int64_t before = c0 * L.bce[1] * L.bce[2];
  if (L.d[0].isc[i0]) {
    before += c1 * L.bce[2];
    if (L.d[1].isc[i1]) before += c2;
  }
  const int64_t flat = ((int64_t)k0 * L.be[1] + k1) * L.be[2] + k2;
  const int64_t b = ((int64_t)b0 * L.bnb[1] + b1) * L.bnb[2] + b2;
  return L.sym_off + b * L.bpb + flat - before;
}

template <typename T>
__device__ __forceinline__ bool all_coarse(const GLevel<T>& L, int i0, int i1, int i2) {
  return g_isc(L.d[0], i0) && g_isc(L.d[1], i1) && g_isc(L.d[2], i2);
}

// Stream position of the coefficient at (i0, i1, i2), flat index `flat`:
// its rank among the level's non-coarse nodes (row-major) plus the level's
// offset and, per index of dimension 0, blk_extra.
template <typename T>
__device__ __forceinline__ int64_t nc_pos(const GLevel<T>& L, int i0, int i1, int i2, int64_t flat) {
  if (L.bmode) return blk_pos(L, i0, i1, i2);
  const int64_t c1 = L.d[1].c, c2 = L.d[2].c;
  int64_t before = (int64_t)g_cb(L.d[0], i0) * c1 * c2;
  if (g_isc(L.d[0], i0)) {
    before += (int64_t)g_cb(L.d[1], i1) * c2;
    if (g_isc(L.d[1], i1)) before += g_cb(L.d[2], i2);
  }
  return L.sym_off + flat - before + (int64_t)i0 * L.blk_extra;
}

// (i0, i1, i2) of a flat node index: divisions by multiplication with the
// extents' rounded-up reciprocals (exact for 32-bit indices), 64-bit divisions
// above them.
struct NodeDiv {
  unsigned n1, n2;
  unsigned long long m1, m2;
  bool wide;
};
inline NodeDiv node_div(int64_t n0, int n1, int n2) {
  NodeDiv d{};
  d.n1 = (unsigned)n1;
  d.n2 = (unsigned)n2;
  d.m1 = ~0ull / d.n1 + 1ull;
  d.m2 = ~0ull / d.n2 + 1ull;
  d.wide = n0 * n1 * n2 > 0xFFFFFFFFll;
  return d;
}
template <typename T>
NodeDiv node_div(const GLevel<T>& L) { return node_div(L.d[0].n, L.d[1].n, L.d[2].n); }
template <typename T>
NodeDiv coarse_div(const GLevel<T>& L) { return node_div(L.d[0].c, L.d[1].c, L.d[2].c); }
// rows i0 of the fine grid, coarse cells of the other two dimensions
template <typename T>
int64_t row_cells(const GLevel<T>& L) { return (int64_t)L.d[0].n * L.d[1].c * L.d[2].c; }
template <typename T>
NodeDiv row_cell_div(const GLevel<T>& L) { return node_div(L.d[0].n, L.d[1].c, L.d[2].c); }
__device__ __forceinline__ void node_of(const NodeDiv& d, int64_t idx, int& i0, int& i1, int& i2) {
  if (!d.wide) {
    const unsigned u = (unsigned)idx;
    const unsigned t = d.n2 == 1u ? u : (unsigned)__umul64hi((unsigned long long)u, d.m2);
    const unsigned q = d.n1 == 1u ? t : (unsigned)__umul64hi((unsigned long long)t, d.m1);
    i2 = (int)(u - t * d.n2);
    i1 = (int)(t - q * d.n1);
    i0 = (int)q;
  } else {
    const int64_t t = idx / d.n2, q = t / d.n1;
    i2 = (int)(idx - t * d.n2);
    i1 = (int)(t - q * d.n1);
    i0 = (int)q;
  }
}

// Coefficients of one global level: D = U - I(U|C) at every node (0 at
// all-coarse nodes, exactly), written to Dfull; the non-coarse ones are
// quantised (mode 0; a histogram pass counts the symbols afterwards) or stored
// (mode 1) at their stream position.  One thread per node: the level's grid is
// small (155^3 at 513^3) and the tables stay in L1, so what counts is enough
// threads in flight and cheap index arithmetic.  (One warp per row of the grid
// took 0.040 ms for the first level at 513^3 against 0.045, and on the few
// long rows of a plane's grid 0.040 against 0.008.)
// With tier != null (the in-cache levels of the block-major grid), the
// quantiser width of a node is rq_ptr[tier[i0] * tstride] (the block's ROI
// tier); otherwise rq_ptr[0].
template <typename T, int MODE>
__global__ void __launch_bounds__(256) gl_fwd_detail(GLevel<T> L, const T* __restrict__ U, T* __restrict__ Dfull,
                                                     uint16_t* sym, int32_t* esc, T* coef, const T* rq_ptr,
                                                     int radius, Scalars* sc, NodeDiv nd,
                                                     const uint8_t* tier = nullptr, int tstride = 0) {
  const GDim<T>&D0 = L.d[0], &D1 = L.d[1], &D2 = L.d[2];
  const int n1 = D1.n, n2 = D2.n;
  const int64_t total = (int64_t)D0.n * n1 * n2;
  const unsigned dict = 2u * (unsigned)radius;
  bool ovf = false;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int i0, i1, i2;
    node_of(nd, idx, i0, i1, i2);
    const int a0 = g_cidx(D0, g_jlo(D0, i0)), b0 = g_cidx(D0, g_jhi(D0, i0));
    const int a1 = g_cidx(D1, g_jlo(D1, i1)), b1 = g_cidx(D1, g_jhi(D1, i1));
    const int a2 = g_cidx(D2, g_jlo(D2, i2)), b2 = g_cidx(D2, g_jhi(D2, i2));
    const T wl0 = g_wl(D0, i0), wr0 = g_wr(D0, i0), wl1 = g_wl(D1, i1), wr1 = g_wr(D1, i1);
    const T wl2 = g_wl(D2, i2), wr2 = g_wr(D2, i2);
    const T* r00 = U + ((int64_t)a0 * n1 + a1) * n2;
    const T* r01 = U + ((int64_t)a0 * n1 + b1) * n2;
    const T* r10 = U + ((int64_t)b0 * n1 + a1) * n2;
    const T* r11 = U + ((int64_t)b0 * n1 + b1) * n2;
    const T ta = fma(wl1, fma(wl2, r00[a2], wr2 * r00[b2]), wr1 * fma(wl2, r01[a2], wr2 * r01[b2]));
    const T tb = fma(wl1, fma(wl2, r10[a2], wr2 * r10[b2]), wr1 * fma(wl2, r11[a2], wr2 * r11[b2]));
    const T e = fma(wl0, ta, wr0 * tb);
    const T dv = U[idx] - e;
    Dfull[idx] = dv;
    if (all_coarse(L, i0, i1, i2)) continue;  // no coefficient
    const int64_t pos = nc_pos(L, i0, i1, i2, idx);
    if (MODE == 0) {
      // the quantiser width of the block's ROI tier (in-cache levels)
      const int64_t tb_ = !tier ? 0 : (int64_t)tier[L.bmode ? blk_of(L, i0, i1, i2) : (int64_t)i0] * tstride;
      const int code = quantize(dv, rq_ptr[tb_], ovf);
      const unsigned u = (unsigned)(code + radius);
      const bool in = u - 1u < dict - 1u;
      const unsigned sv = in ? u : 0u;
      sym[pos] = (uint16_t)sv;
      if (!in) esc[pos] = code;
    } else {
      coef[pos] = dv;
    }
  }
  if (MODE == 0 && ovf) atomicOr(&sc->status, ST_OVERFLOW);
}

// The same with a warp per grid row (i0, i1), whose interpolation sources,
// weights and stream offset are taken once, the lanes walking i2.
template <typename T, int MODE>
__global__ void __launch_bounds__(256) gl_fwd_detail_rows(GLevel<T> L, const T* __restrict__ U,
                                                          T* __restrict__ Dfull, uint16_t* sym, int32_t* esc, T* coef,
                                                          const T* rq_ptr, int radius, Scalars* sc,
                                                          const uint8_t* tier, int tstride) {
  const GDim<T>&D0 = L.d[0], &D1 = L.d[1], &D2 = L.d[2];
  const int n1 = D1.n, n2 = D2.n;
  const int64_t rows = (int64_t)D0.n * n1, c12 = (int64_t)D1.c * D2.c;
  const unsigned dict = 2u * (unsigned)radius;
  bool ovf = false;
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < rows; row += nwarps) {
    const int i0 = (int)(row / n1), i1 = (int)(row - (int64_t)i0 * n1);
    const T rq_row = MODE == 0 && !L.bmode ? rq_ptr[tier ? (int)tier[i0] * tstride : 0] : T(0);
    const int a0 = g_cidx(D0, g_jlo(D0, i0)), b0 = g_cidx(D0, g_jhi(D0, i0));
    const int a1 = g_cidx(D1, g_jlo(D1, i1)), b1 = g_cidx(D1, g_jhi(D1, i1));
    const T wl0 = g_wl(D0, i0), wr0 = g_wr(D0, i0), wl1 = g_wl(D1, i1), wr1 = g_wr(D1, i1);
    const T* r00 = U + ((int64_t)a0 * n1 + a1) * n2;
    const T* r01 = U + ((int64_t)a0 * n1 + b1) * n2;
    const T* r10 = U + ((int64_t)b0 * n1 + a1) * n2;
    const T* r11 = U + ((int64_t)b0 * n1 + b1) * n2;
    const bool cc01 = g_isc(D0, i0) && g_isc(D1, i1);  // the row holds all-coarse nodes
    // stream rank of the row's first node: flat index minus the all-coarse nodes before it
    int64_t before = (int64_t)g_cb(D0, i0) * c12;
    if (g_isc(D0, i0)) before += (int64_t)g_cb(D1, i1) * D2.c;
    const int64_t rbase = L.sym_off + row * n2 - before + (int64_t)i0 * L.blk_extra;
    for (int i2 = lane; i2 < n2; i2 += 32) {
      const int a2 = g_cidx(D2, g_jlo(D2, i2)), b2 = g_cidx(D2, g_jhi(D2, i2));
      const T wl2 = g_wl(D2, i2), wr2 = g_wr(D2, i2);
      const T ta = fma(wl1, fma(wl2, r00[a2], wr2 * r00[b2]), wr1 * fma(wl2, r01[a2], wr2 * r01[b2]));
      const T tb = fma(wl1, fma(wl2, r10[a2], wr2 * r10[b2]), wr1 * fma(wl2, r11[a2], wr2 * r11[b2]));
      const T e = fma(wl0, ta, wr0 * tb);
      const int64_t idx = row * n2 + i2;
      const T dv = U[idx] - e;
      Dfull[idx] = dv;
      if (cc01 && g_isc(D2, i2)) continue;  // all-coarse node: no coefficient
      int64_t pos;
      T rq = rq_row;
      if (L.bmode) {  // block-major order; the block's ROI tier
        pos = blk_pos(L, i0, i1, i2);
        if (MODE == 0) rq = rq_ptr[tier ? (int)tier[blk_of(L, i0, i1, i2)] * tstride : 0];
      } else {
        pos = rbase + i2 - (cc01 ? g_cb(D2, i2) : 0);
      }
      if (MODE == 0) {
        const int code = quantize(dv, rq, ovf);
        const unsigned u = (unsigned)(code + radius);
        const bool in = u - 1u < dict - 1u;
        const unsigned sv = in ? u : 0u;
        sym[pos] = (uint16_t)sv;
        if (!in) esc[pos] = code;
      } else {
        coef[pos] = dv;
      }
    }
  }
  if (MODE == 0 && ovf) atomicOr(&sc->status, ST_OVERFLOW);
}

// Whether a warp a row pays: single precision, long rows, and enough of them for
// many steps of every warp (the two levels of 400x410x390, B = 8, with the line
// passes: 2350 us against 2595; of 100x90x80 85 against 82, of 300x290x310 doubles
// 3334 against 3226).
template <typename T>
bool detail_by_rows(const GLevel<T>& L, int nsm) {
  return sizeof(T) == 4 && L.d[2].n >= 64 && (int64_t)L.d[0].n * L.d[1].n >= 256ll * nsm;
}

// One restriction pass of a global level as a dense contraction with the
// level's projection P = M_c^{-1} I^T M_f (c x n) along dimension DIM:
//   out[b][J][col] = sum_i P[J][i] in[b][i][col]
// (the same operator as band products followed by the tridiagonal solve).
// A CTA owns 64 columns of one batch; 32 x 64 tiles of `in` (its unit-stride
// index varying fastest across threads) and 32 x 32 tiles of P are staged in
// shared memory; a thread keeps 8 outputs of each 32-row tile of J.
//   DIM 2: in (n0,n1,n2) -> out (n0,n1,c2), columns = lines (n0*n1)
//   DIM 1: in (n0,n1,c2) -> out (n0,c1,c2), batches i0, columns j2
//   DIM 0: in (n0,c1,c2) -> out (c0,c1,c2), columns (j1,j2); FINAL 1: out =
//          U|C + z (forward), FINAL 2: out = U - z (inverse, U compact)
struct ApplyShape {
  int64_t nb, ncol;
  int64_t in_b, in_i, in_c;
  int64_t out_b, out_j, out_c;
};

template <typename T>
ApplyShape apply_shape(const GLevel<T>& L, int dim) {
  const int64_t n0 = L.d[0].n, n1 = L.d[1].n, n2 = L.d[2].n, c1 = L.d[1].c, c2 = L.d[2].c;
  ApplyShape S{};
  if (dim == 2) {
    S.nb = 1; S.ncol = n0 * n1; S.in_i = 1; S.in_c = n2; S.out_j = 1; S.out_c = c2;
  } else if (dim == 1) {
    S.nb = n0; S.ncol = c2; S.in_b = n1 * c2; S.in_i = c2; S.in_c = 1; S.out_b = c1 * c2; S.out_j = c2; S.out_c = 1;
  } else {
    S.nb = 1; S.ncol = c1 * c2; S.in_i = c1 * c2; S.in_c = 1; S.out_j = c1 * c2; S.out_c = 1;
  }
  return S;
}

constexpr int kApplyCols = 64, kApplyK = 32, kApplyJ = 32;

template <typename T, int DIM, int FINAL>
__global__ void __launch_bounds__(256) gl_apply(GLevel<T> L, ApplyShape S, const T* __restrict__ in,
                                                T* __restrict__ out, const T* __restrict__ U) {
  __shared__ T s_in[kApplyK][kApplyCols + 1];
  __shared__ T s_p[kApplyJ][kApplyK + 1];
  const GDim<T>& D = L.d[DIM];
  const int n = D.n, c = D.c;
  const int64_t tiles = (S.ncol + kApplyCols - 1) / kApplyCols;
  const int64_t b = blockIdx.x / tiles;
  const int64_t col0 = (blockIdx.x - b * tiles) * kApplyCols;
  const int tid = threadIdx.x, tc = tid & (kApplyCols - 1), jg = tid >> 6;
  const T* inb = in + b * S.in_b;
  const bool unit_i = S.in_i == 1;
  for (int jt = 0; jt < c; jt += kApplyJ) {
    T acc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[q] = T(0);
    for (int i0 = 0; i0 < n; i0 += kApplyK) {
      __syncthreads();  // the previous tile has been consumed
#pragma unroll
      for (int r = 0; r < kApplyK * kApplyCols / 256; ++r) {
        const int e = tid + 256 * r;
        const int ii = unit_i ? (e & (kApplyK - 1)) : (e >> 6);
        const int cc = unit_i ? (e >> 5) : (e & (kApplyCols - 1));
        const int64_t col = col0 + cc;
        T v = T(0);
        if (i0 + ii < n && col < S.ncol) v = inb[(int64_t)(i0 + ii) * S.in_i + col * S.in_c];
        s_in[ii][cc] = v;
      }
#pragma unroll
      for (int r = 0; r < kApplyJ * kApplyK / 256; ++r) {
        const int e = tid + 256 * r, ii = e & (kApplyK - 1), jj = e >> 5;
        s_p[jj][ii] = (jt + jj < c && i0 + ii < n) ? D.P[(int64_t)(jt + jj) * n + i0 + ii] : T(0);
      }
      __syncthreads();
#pragma unroll 8
      for (int ii = 0; ii < kApplyK; ++ii) {
        const T x = s_in[ii][tc];
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[q] = fma(s_p[jg * 8 + q][ii], x, acc[q]);
      }
    }
    const int64_t col = col0 + tc;
    if (col < S.ncol) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int J = jt + jg * 8 + q;
        if (J >= c) break;
        const int64_t o = b * S.out_b + (int64_t)J * S.out_j + col * S.out_c;
        if (FINAL == 1) {
          const int c2 = L.d[2].c, j1 = (int)(col / c2), j2 = (int)(col - (int64_t)j1 * c2);
          const int64_t u = ((int64_t)L.d[0].cidx[J] * L.d[1].n + L.d[1].cidx[j1]) * L.d[2].n + L.d[2].cidx[j2];
          out[o] = U[u] + acc[q];
        } else if (FINAL == 2) {
          out[o] = U[o] - acc[q];
        } else {
          out[o] = acc[q];
        }
      }
    }
  }
}

// One restriction pass of a global level, line by line along dimension DIM:
// r = I^T M_f d (five-point band), then M_c z = r by the Thomas recurrences,
// each evaluated as a warp scan of affine maps (lane l owns the E coarse rows
// l*E .. l*E+E-1, composes their maps, combines them across the warp with
// shuffles, then replays its rows from the combined input).  The same
// operator as the dense projection in gl_apply, in O(n) work per line.
// A CTA stages 2^LSH lines (line_tile_shift) in shared memory,
// read coalesced along the line when it is contiguous (DIM 2) and across the
// lines otherwise; eight warps take one line at a time.  Shapes and FINAL as
// for gl_apply.  E is odd, so the lanes' rows of a segment never share a bank.
// Lines of a CTA, as a shift: a 128-byte row of columns, or a 32-byte sector
// when those tiles would leave SMs idle (a plane's 455 lines of 605 nodes in 15
// CTAs of 32 lines took 24 us, in 57 of 8 14).
template <typename T>
constexpr int line_full_shift() { return sizeof(T) == 4 ? 5 : 4; }
template <typename T>
int line_tile_shift(int64_t nb, int64_t ncol, int nsm) {
  constexpr int full = line_full_shift<T>();
  return nb * ((ncol >> full) + 1) < 2 * nsm ? full - 2 : full;
}
inline int line_segment(int c) {  // rows per lane (0: the line is too long for gl_line)
  const int e = (c + 31) / 32;
  return e <= 1 ? 1 : e <= 3 ? 3 : e <= 9 ? 9 : e <= 17 ? 17 : 0;
}
// Whether a level's coefficients are taken by its first restriction pass: where
// that pass's lines fill the SMs (a plane's 455 lines of 605 nodes: 38 us in
// one kernel, 8 + 14.4 in two; 155^3: 53 in one, 45 + 18 in two, and for the
// inverse 27 against 22 + 18).
template <typename T>
bool coefs_in_line_pass(const GLevel<T>& L, int nsm) {
  const int64_t lines = (int64_t)L.d[0].n * L.d[1].n;
  return line_segment(L.d[2].c) && lines >> line_tile_shift<T>(1, lines, nsm) >= nsm;
}
template <typename T>
size_t line_smem(int n, int c, int lsh) {
  return ((size_t)((n | 1) + (c | 1)) << lsh) * sizeof(T);
}

// z = M_c^-1 r of one line in shared memory, in place, by a warp.  AGAIN: times
// that the lanes replay their rows once more, from the value their neighbour
// computed; each time a value's roundings are those of the serial recurrence
// E rows further back.
template <typename T, int E, int AGAIN = 0>
__device__ __forceinline__ void line_scan_solve(const GDim<T>& D, T* r, const int lane) {
  const int c = D.c;
  const int j0 = lane * E;
  T y[E];
  // forward recurrence y_J = r_J - tm_J y_{J-1} (y_{-1} = 0)
  T a = T(0), m = T(1);
#pragma unroll
  for (int k = 0; k < E; ++k) {
    const int J = j0 + k;
    if (J < c) {
      const T t = D.tm[J];
      a = fma(-t, a, r[J]);
      m = -t * m;
    }
  }
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const T pa = __shfl_up_sync(0xffffffffu, a, off), pm = __shfl_up_sync(0xffffffffu, m, off);
    if (lane >= off) {
      a = fma(m, pa, a);
      m *= pm;
    }
  }
  T prev = __shfl_up_sync(0xffffffffu, a, 1);
  if (lane == 0) prev = T(0);
#pragma unroll
  for (int p = 0; p <= AGAIN; ++p) {
#pragma unroll
    for (int k = 0; k < E; ++k) {
      const int J = j0 + k;
      if (J < c) {
        y[k] = fma(-D.tm[J], prev, r[J]);
        prev = y[k];
      }
    }
    if (p < AGAIN) {
      prev = __shfl_up_sync(0xffffffffu, prev, 1);
      if (lane == 0) prev = T(0);
    }
  }
  // backward recurrence z_J = (y_J - tsup_J z_{J+1}) tib_J (z_c = 0)
  a = T(0);
  m = T(1);
#pragma unroll
  for (int k = E - 1; k >= 0; --k) {
    const int J = j0 + k;
    if (J < c) {
      const T ib = D.tib[J], q = -D.tsup[J] * ib;
      a = fma(q, a, y[k] * ib);
      m = q * m;
    }
  }
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const T pa = __shfl_down_sync(0xffffffffu, a, off), pm = __shfl_down_sync(0xffffffffu, m, off);
    if (lane + off < 32) {
      a = fma(m, pa, a);
      m *= pm;
    }
  }
  T next = __shfl_down_sync(0xffffffffu, a, 1);
  if (lane == 31) next = T(0);
  __syncwarp();  // every lane has read its r before any z overwrites it
#pragma unroll
  for (int p = 0; p <= AGAIN; ++p) {
#pragma unroll
    for (int k = E - 1; k >= 0; --k) {
      const int J = j0 + k;
      if (J < c) {
        next = fma(-D.tsup[J], next, y[k]) * D.tib[J];
        if (p == AGAIN) r[J] = next;
      }
    }
    if (p < AGAIN) {  // (a lane without rows holds 0)
      next = __shfl_down_sync(0xffffffffu, next, 1);
      if (lane == 31) next = T(0);
    }
  }
}

// What the first (DIM 2) pass of a global level restricts: a grid in memory
// (SRC_GRID); the level's coefficients, computed from the grid U and quantised
// (SRC_CODE) or stored (SRC_COEF) at their stream position as the lines are
// staged; the coefficients read back from the stream's codes (SRC_DECODE) or
// values (SRC_READ), kept in the grid D for the interpolation.
enum { SRC_GRID = 0, SRC_CODE = 1, SRC_COEF = 2, SRC_DECODE = 3, SRC_READ = 4 };
template <typename T>
struct LineSrc {
  uint16_t* sym;
  int32_t* esc;
  T* coef;
  const T* rq;      // SRC_CODE: the level's reciprocal bin width
  const double* q;  // SRC_DECODE: its bin width
  T* D;
  int radius;
  Scalars* sc;
};

// Stages line `line` (its row of U at u) of a global level by a warp: the same
// operations per node as gl_fwd_detail and gl_inv_dequant, with everything
// that depends on (i0, i1) taken once a line.  Bound by issue and the latency
// of a warp's loads; four nodes of a lane in flight were slower (0.060 against
// 0.053 ms at 155^3: the lines are five nodes a lane, the rest is thrown away).
template <typename T, int SRC>
__device__ __forceinline__ void stage_coefs(const GLevel<T>& L, const LineSrc<T>& W, const T* __restrict__ U,
                                            int64_t line, T* x, int lane, bool& ovf) {
  const GDim<T>&D0 = L.d[0], &D1 = L.d[1], &D2 = L.d[2];
  const int n1 = D1.n, n2 = D2.n;
  const int i0 = (int)(line / n1), i1 = (int)(line - (int64_t)i0 * n1);
  const bool ic0 = g_isc(D0, i0), cc = ic0 && g_isc(D1, i1);
  int64_t before = (int64_t)g_cb(D0, i0) * D1.c * D2.c;
  if (ic0) before += (int64_t)g_cb(D1, i1) * D2.c;
  const int64_t flat = line * n2, pos0 = L.sym_off + flat - before;
  if (SRC == SRC_CODE || SRC == SRC_COEF) {
    const int a0 = g_cidx(D0, g_jlo(D0, i0)), b0 = g_cidx(D0, g_jhi(D0, i0));
    const int a1 = g_cidx(D1, g_jlo(D1, i1)), b1 = g_cidx(D1, g_jhi(D1, i1));
    const T wl0 = g_wl(D0, i0), wr0 = g_wr(D0, i0), wl1 = g_wl(D1, i1), wr1 = g_wr(D1, i1);
    const T* r00 = U + ((int64_t)a0 * n1 + a1) * n2;
    const T* r01 = U + ((int64_t)a0 * n1 + b1) * n2;
    const T* r10 = U + ((int64_t)b0 * n1 + a1) * n2;
    const T* r11 = U + ((int64_t)b0 * n1 + b1) * n2;
    const T rq = SRC == SRC_CODE ? *W.rq : T(0);
    const unsigned dict = 2u * (unsigned)W.radius;
    for (int i2 = lane; i2 < n2; i2 += 32) {
      const int a2 = g_cidx(D2, g_jlo(D2, i2)), b2 = g_cidx(D2, g_jhi(D2, i2));
      const T wl2 = g_wl(D2, i2), wr2 = g_wr(D2, i2);
      const T ta = fma(wl1, fma(wl2, r00[a2], wr2 * r00[b2]), wr1 * fma(wl2, r01[a2], wr2 * r01[b2]));
      const T tb = fma(wl1, fma(wl2, r10[a2], wr2 * r10[b2]), wr1 * fma(wl2, r11[a2], wr2 * r11[b2]));
      const T e = fma(wl0, ta, wr0 * tb);
      const T dv = U[flat + i2] - e;
      x[i2] = dv;
      if (cc && g_isc(D2, i2)) continue;  // no coefficient
      const int64_t pos = pos0 + i2 - (cc ? g_cb(D2, i2) : 0);
      if (SRC == SRC_CODE) {
        const int code = quantize(dv, rq, ovf);
        const unsigned u = (unsigned)(code + W.radius);
        const bool in = u - 1u < dict - 1u;
        const unsigned sv = in ? u : 0u;
        W.sym[pos] = (uint16_t)sv;
        if (!in) W.esc[pos] = code;
      } else {
        W.coef[pos] = dv;
      }
    }
  } else {
    const T q = SRC == SRC_DECODE ? (T)*W.q : T(0);
    for (int i2 = lane; i2 < n2; i2 += 32) {
      T v = T(0);
      if (!(cc && g_isc(D2, i2))) {
        const int64_t pos = pos0 + i2 - (cc ? g_cb(D2, i2) : 0);
        if (SRC == SRC_DECODE) {
          const unsigned s = W.sym[pos];
          v = dequant(s ? (int)s - W.radius : W.esc[pos], q);
        } else {
          v = W.coef[pos];
        }
      }
      x[i2] = v;
      W.D[flat + i2] = v;
    }
  }
}

template <typename T, int DIM, int FINAL, int E, int SRC, int LSH>
__global__ void __launch_bounds__(256) gl_line(GLevel<T> L, ApplyShape S, const T* __restrict__ in,
                                               T* __restrict__ out, const T* __restrict__ U, LineSrc<T> W) {
  // lines of the CTA (with the shift an argument, the short lines of a block-major
  // grid, 8 nodes and 5 columns of 47,000 blocks, took 93 us against 75)
  constexpr int lsh = LSH, LT = 1 << LSH;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const GDim<T>& D = L.d[DIM];
  const int n = D.n, c = D.c, sn = n | 1, sc = c | 1;
  T* s_in = reinterpret_cast<T*>(smem_raw);  // [LT][sn] the lines
  T* s_out = s_in + LT * sn;                  // [LT][sc] r, then z
  const int64_t tiles = (S.ncol + LT - 1) / LT;
  const int64_t b = blockIdx.x / tiles;
  const int64_t col0 = (blockIdx.x - b * tiles) * LT;
  const int nl = (int)(S.ncol - col0 < LT ? S.ncol - col0 : LT);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const T* inb = in + b * S.in_b;
  if (SRC != SRC_GRID) {
    bool ovf = false;
    for (int w = warp; w < nl; w += 8) stage_coefs<T, SRC>(L, W, in, col0 + w, s_in + w * sn, lane, ovf);
    if (SRC == SRC_CODE && ovf) atomicOr(&W.sc->status, ST_OVERFLOW);
  } else if (S.in_i == 1) {
    for (int w = warp; w < nl; w += 8)
      for (int i = lane; i < n; i += 32) s_in[w * sn + i] = inb[(col0 + w) * S.in_c + i];
  } else {
    for (int e = threadIdx.x; e < n * LT; e += 256) {
      const int i = e >> lsh, w = e - (i << lsh);
      if (w < nl) s_in[w * sn + i] = inb[(int64_t)i * S.in_i + (col0 + w) * S.in_c];
    }
  }
  __syncthreads();
  for (int w = warp; w < nl; w += 8) {
    const T* x = s_in + w * sn;
    T* r = s_out + w * sc;
    if (c == n) {  // a dimension of at most two nodes is not coarsened
      for (int J = lane; J < c; J += 32) r[J] = x[J];
      continue;
    }
    for (int J = lane; J < c; J += 32) {
      const int f = D.f0[J];
      T v = T(0);
#pragma unroll
      for (int m = 0; m < 5; ++m)
        if (f + m < n) v = fma(D.band[5 * J + m], x[f + m], v);
      r[J] = v;
    }
    __syncwarp();
    line_scan_solve<T, E>(D, r, lane);
  }
  __syncthreads();
  auto emit = [&](int J, int w) {
    const int64_t col = col0 + w;
    const int64_t o = b * S.out_b + (int64_t)J * S.out_j + col * S.out_c;
    const T z = s_out[w * sc + J];
    if (FINAL == 1) {  // (j0, j1, j2): (J, col) along dimension 0, (b, J, col) along dimension 1
      const int c2 = L.d[2].c, j1 = DIM == 1 ? J : (int)(col / c2), j2 = (int)(DIM == 1 ? col : col - (int64_t)j1 * c2);
      const int j0 = DIM == 1 ? (int)b : J;
      const int64_t u = ((int64_t)L.d[0].cidx[j0] * L.d[1].n + L.d[1].cidx[j1]) * L.d[2].n + L.d[2].cidx[j2];
      out[o] = U[u] + z;
    } else if (FINAL == 2) {
      out[o] = U[o] - z;
    } else {
      out[o] = z;
    }
  };
  if (S.out_j == 1) {
    for (int w = warp; w < nl; w += 8)
      for (int J = lane; J < c; J += 32) emit(J, w);
  } else {
    for (int e = threadIdx.x; e < c * LT; e += 256) {
      const int J = e >> lsh, w = e - (J << lsh);
      if (w < nl) emit(J, w);
    }
  }
}

// The restriction pass along an identity dimension 0 (the block index of
// the block-major grid): z = in, elementwise, with FINAL as for gl_apply
// (1: out = U|C + z; 2: out = U - z; 0: out = z).  in, out: (n0, c1, c2).
template <typename T, int FINAL>
__global__ void __launch_bounds__(256) gl_ident0(GLevel<T> L, const T* __restrict__ in, T* __restrict__ out,
                                                 const T* __restrict__ U) {
  const int n0 = L.d[0].n, c1 = L.d[1].c, c2 = L.d[2].c, n1 = L.d[1].n, n2 = L.d[2].n;
  const int64_t total = (int64_t)n0 * c1 * c2;
  for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < total; o += (int64_t)gridDim.x * blockDim.x) {
    const T z = in[o];
    if (FINAL == 1) {
      const int j2 = (int)(o % c2);
      const int64_t t = o / c2;
      const int j1 = (int)(t % c1);
      const int i0 = (int)(t / c1);
      out[o] = U[((int64_t)i0 * n1 + g_cidx(L.d[1], j1)) * n2 + g_cidx(L.d[2], j2)] + z;
    } else if (FINAL == 2) {
      out[o] = U[o] - z;
    } else {
      out[o] = z;
    }
  }
}

// Between a grid and its blocks in block-major order: block b (row-major
// over the block grid nb) of edges e[3] (1 along dimensions of extent 1) is
// stored as a contiguous E1 x E2 tile, its axes the grid dimensions ax[0] and
// ax[1] (ax[0] = -1: E1 = 1).  DIR 0 gathers (nodes outside the grid read as
// zero), DIR 1 scatters the nodes inside the grid.
struct Reblock {
  int64_t g[3];   // grid shape
  int e[3];       // block edge per dimension
  int nb[3];      // blocks per dimension
  int ax[2];      // grid dimension of tile axis 1 and 2 (-1: none)
  int E1, E2;     // tile extents
  int64_t nblk;
};

template <typename T, int DIR>
__global__ void __launch_bounds__(256) reblock_kernel(Reblock R, T* __restrict__ grid, T* __restrict__ blocked) {
  const int64_t total = R.nblk * R.E1 * R.E2;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int k2 = (int)(idx % R.E2);
    const int64_t t = idx / R.E2;
    const int k1 = (int)(t % R.E1);
    const int64_t b = t / R.E1;
    const int b2 = (int)(b % R.nb[2]);
    const int64_t t2 = b / R.nb[2];
    const int b1 = (int)(t2 % R.nb[1]);
    const int b0 = (int)(t2 / R.nb[1]);
    int64_t c[3] = {(int64_t)b0 * R.e[0], (int64_t)b1 * R.e[1], (int64_t)b2 * R.e[2]};
    if (R.ax[0] >= 0) c[R.ax[0]] += k1;
    c[R.ax[1]] += k2;
    const bool in = c[0] < R.g[0] && c[1] < R.g[1] && c[2] < R.g[2];
    const int64_t gi = (c[0] * R.g[1] + c[1]) * R.g[2] + c[2];
    if (DIR == 0) blocked[idx] = in ? grid[gi] : T(0);
    else if (in) grid[gi] = blocked[idx];
  }
}

// Between a grid of shape S and its zero-padded copy of shape P (P >= S per
// dimension, the padding at the high end): DIR 0 pads (dst = padded),
// DIR 1 crops (dst = the grid).
template <typename T, int DIR>
__global__ void __launch_bounds__(256) pad_kernel(const T* __restrict__ src, T* __restrict__ dst, int64_t s0,
                                                  int64_t s1, int64_t s2, int64_t p0, int64_t p1, int64_t p2) {
  const int64_t total = DIR == 0 ? p0 * p1 * p2 : s0 * s1 * s2;
  const int64_t n1 = DIR == 0 ? p1 : s1, n2 = DIR == 0 ? p2 : s2;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i2 = idx % n2, t = idx / n2, i1 = t % n1, i0 = t / n1;
    if (DIR == 0) dst[idx] = (i0 < s0 && i1 < s1 && i2 < s2) ? src[(i0 * s1 + i1) * s2 + i2] : T(0);
    else dst[idx] = src[(i0 * p1 + i1) * p2 + i2];
  }
}

// Inverse: dequantised coefficients into a full grid (0 at all-coarse nodes).
// (With 64-bit divisions for the node's indices it took 0.027 ms for the first
// level at 513^3 against 0.022.)
// With tier != null (the in-cache levels of the block-major grid), the
// quantiser width of the nodes with index i0 is q_ptr[tier[i0] * tstride];
// the tier byte is range-checked against ntiers (a corrupt stream flags sc).
template <typename T, int MODE>
__global__ void gl_inv_dequant(GLevel<T> L, const uint16_t* __restrict__ sym, const int32_t* __restrict__ esc,
                               const T* __restrict__ coef, const double* q_ptr, int radius, T* __restrict__ Dfull,
                               NodeDiv nd, const uint8_t* tier = nullptr, int tstride = 0, int ntiers = 1,
                               Scalars* sc = nullptr) {
  const int64_t total = (int64_t)L.d[0].n * L.d[1].n * L.d[2].n;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int i0, i1, i2;
    node_of(nd, idx, i0, i1, i2);
    T v = T(0);
    if (!all_coarse(L, i0, i1, i2)) {
      const int64_t pos = nc_pos(L, i0, i1, i2, idx);
      int tr = tier ? (int)tier[L.bmode ? blk_of(L, i0, i1, i2) : (int64_t)i0] : 0;
      if (tr >= ntiers) {
        if (sc) atomicOr(&sc->status, ST_CORRUPT);
        tr = 0;
      }
      const T q = MODE == 0 ? (T)q_ptr[tr * tstride] : T(0);
      if (MODE == 0) {
        const unsigned s = sym[pos];
        const int code = s ? (int)s - radius : esc[pos];
        v = dequant(code, q);
      } else {
        v = coef[pos];
      }
    }
    Dfull[idx] = v;
  }
}

// Inverse: U = I(Uc) + D in place (Dfull holds D on entry, U on exit).  One
// thread per pair of coarse cells' rows: the up to four nodes of row i0 that
// follow coarse nodes J1, J2 (each, and the node after it where that is not
// coarse) share the corner values and the partial interpolants.  A coarse node
// interpolates from itself with weights 1 and 0.  A thread per node, with the
// tables and all eight values read for each, took 0.029 ms for the first level
// at 513^3 (155^3 nodes) and 0.007 for the second against 0.020 and 0.007; a
// thread per cell in all three dimensions 0.026 and 0.011.
template <typename T>
__global__ void __launch_bounds__(256) gl_inv_interp(GLevel<T> L, const T* __restrict__ Uc, T* __restrict__ Dfull,
                                                     NodeDiv cd) {
  const GDim<T>&D0 = L.d[0], &D1 = L.d[1], &D2 = L.d[2];
  const int c1 = D1.c, c2 = D2.c, n1 = D1.n, n2 = D2.n;
  const int64_t total = (int64_t)D0.n * c1 * c2;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    int i0, J1, J2;
    node_of(cd, e, i0, J1, J2);
    const int a0 = g_jlo(D0, i0), b0 = g_jhi(D0, i0), i1 = g_cidx(D1, J1), i2 = g_cidx(D2, J2);
    const T wl0 = g_wl(D0, i0), wr0 = g_wr(D0, i0);
    const bool f1 = i1 + 1 < n1 && !g_isc(D1, i1 + 1), f2 = i2 + 1 < n2 && !g_isc(D2, i2 + 1);
    T* const u = Dfull + ((int64_t)i0 * n1 + i1) * n2 + i2;
    T d[2][2];
#pragma unroll
    for (int k1 = 0; k1 < 2; ++k1)
#pragma unroll
      for (int k2 = 0; k2 < 2; ++k2) d[k1][k2] = (!k1 || f1) && (!k2 || f2) ? u[(int64_t)k1 * n2 + k2] : T(0);
    const T wl1 = f1 ? D1.wl[i1 + 1] : T(1), wr1 = f1 ? D1.wr[i1 + 1] : T(0);
    const T wl2 = f2 ? D2.wl[i2 + 1] : T(1), wr2 = f2 ? D2.wr[i2 + 1] : T(0);
    // the nodes (k1, k2) interpolated along dimensions 2 and 1 in coarse row x0
    auto plane = [&](int x0, T (&t)[2][2]) {
      const T* r0 = Uc + ((int64_t)x0 * c1 + J1) * c2 + J2;
      const T* r1 = f1 ? r0 + c2 : r0;
      const T g00 = r0[0], g01 = f2 ? r0[1] : g00, g10 = r1[0], g11 = f2 ? r1[1] : g10;
      const T s00 = fma(T(1), g00, T(0) * g00), s01 = fma(wl2, g00, wr2 * g01);
      const T s10 = fma(T(1), g10, T(0) * g10), s11 = fma(wl2, g10, wr2 * g11);
      t[0][0] = fma(T(1), s00, T(0) * s00);
      t[0][1] = fma(T(1), s01, T(0) * s01);
      t[1][0] = fma(wl1, s00, wr1 * s10);
      t[1][1] = fma(wl1, s01, wr1 * s11);
    };
    T ta[2][2], tb[2][2];
    plane(a0, ta);
    plane(b0, tb);
#pragma unroll
    for (int k1 = 0; k1 < 2; ++k1)
#pragma unroll
      for (int k2 = 0; k2 < 2; ++k2)
        if ((!k1 || f1) && (!k2 || f2))
          u[(int64_t)k1 * n2 + k2] = fma(wl0, ta[k1][k2], wr0 * tb[k1][k2]) + d[k1][k2];
  }
}

// Coarsest array: quantised directly (mode 0) or stored (mode 1).
template <typename T, int MODE>
__global__ void coarsest_fwd(const T* __restrict__ U, int64_t count, int64_t sym_off, uint16_t* sym, int32_t* esc,
                             T* coef, const T* rq_ptr, int radius, Scalars* sc) {
  const T rq = MODE == 0 ? *rq_ptr : T(0);
  bool ovf = false;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
    if (MODE == 0) {
      const int code = quantize(U[i], rq, ovf);
      const bool in = code > -radius && code < radius;
      const unsigned sv = in ? (unsigned)(code + radius) : 0u;
      sym[sym_off + i] = (uint16_t)sv;
      if (!in) esc[sym_off + i] = code;
    } else {
      coef[sym_off + i] = U[i];
    }
  }
  if (MODE == 0 && ovf) atomicOr(&sc->status, ST_OVERFLOW);
}

template <typename T, int MODE>
__global__ void coarsest_inv(T* __restrict__ U, int64_t count, int64_t sym_off, const uint16_t* sym, const int32_t* esc,
                             const T* coef, const double* q_ptr, int radius) {
  const T q = MODE == 0 ? (T)*q_ptr : T(0);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
    if (MODE == 0) {
      const unsigned s = sym[sym_off + i];
      const int code = s ? (int)s - radius : esc[sym_off + i];
      U[i] = dequant(code, q);
    } else {
      U[i] = coef[sym_off + i];
    }
  }
}

}  // namespace bm
